"""The tensor-core attention kernel where its tiles and pages end: pages that its key block does not divide, pages
shorter than one block, query tiles with one row, head dimension 32, windows of one block and of several splits, more
items than CTAs, and scores that rise along the keys, away from the first ones, which are a row's reference."""
import numpy as np
import pytest

from oracle import nfd_oracle as O
from paper_2506_01380_b200 import inputs as I

pytestmark = pytest.mark.gpu

# bf16 inputs and outputs: the error is that of rounding the output (1.7e-3 relative for normal data; held to that in
# test_gpu_attention_values.py); the bounds here are those of the other bf16 cases.
TOL_ABS, TOL_REL = 3e-2, 1e-2


# (latent_h, latent_w) with patch 2 -> tokens per frame h*w/4
@pytest.mark.parametrize("hw,head_dim,heads,n_kv,n_q,window,rise", [
    ((8, 6), 64, 4, 20, 4, 16, 0),        # 12 tokens: a page is a fraction of a block
    ((16, 16), 64, 4, 17, 1, 16, 0),      # 64: the smallest block divides the page
    ((26, 10), 64, 4, 3, 2, 2, 0),        # 65: one key and one query row beyond 64
    ((254, 2), 64, 2, 3, 1, 2, 0),        # 127
    ((32, 16), 64, 2, 3, 1, 2, 0),        # 128: exactly one query tile
    ((86, 6), 64, 2, 4, 2, 3, 0),         # 129: a query tile of one row
    ((40, 22), 64, 16, 12, 3, 9, 0),      # 220: several items per CTA
    ((48, 28), 64, 16, 40, 8, 32, 0),     # 336
    ((48, 28), 64, 4, 17, 1, 16, 1),
    ((40, 22), 64, 4, 17, 4, 16, 1),
    ((16, 16), 32, 4, 6, 2, 4, 0),        # head dimension 32
    ((26, 14), 32, 12, 9, 2, 5, 1),       # 91
])
def test_pages_and_tiles(hw, head_dim, heads, n_kv, n_q, window, rise):
    import torch
    from paper_2506_01380_b200.nfd import NFD
    rope = dict(rope_t=16, rope_h=24, rope_w=24) if head_dim == 64 else dict(rope_t=8, rope_h=12, rope_w=12)
    cfg = I.make_cfg("nfd310m", n_layers=1, d_model=heads * head_dim, n_heads=heads, head_dim=head_dim, d_mlp=256,
                     latent_h=hw[0], latent_w=hw[1], ctx_frames=window, max_spec=8, **rope)
    T = I.tokens_per_frame(cfg)
    g = NFD(cfg, I.make_weights(cfg, 0))
    q, k, v = I.make_qkv(heads, head_dim, n_q * T, n_kv * T, seed=T + head_dim)
    if rise:
        k = k * np.repeat(2.0 ** np.minimum(np.arange(n_kv), 5), T).astype(np.float32)[None, :, None]
    t = [torch.as_tensor(a).cuda().bfloat16() for a in (q, k, v)]
    out = g.attention(*t, n_q, n_kv, window)
    again = g.attention(*t, n_q, n_kv, window)
    assert torch.equal(out, again)
    ref = O.attention_block_causal(q, k, v, np.repeat(np.arange(n_kv - n_q, n_kv), T), np.repeat(np.arange(n_kv), T),
                                   window).transpose(1, 0, 2).reshape(n_q * T, heads * head_dim)
    got = out.float().cpu().numpy().astype(np.float64)
    assert np.all(np.isfinite(got))
    assert np.abs(got - ref).max() <= TOL_ABS
    assert np.linalg.norm(got - ref) / np.linalg.norm(ref) <= TOL_REL
    assert g.status() == 0


@pytest.mark.parametrize("kind,heads,T,dh,n_kv,n_q,window", [
    ("bf16", 3, 77, 32, 9, 2, 5), ("bf16", 5, 129, 64, 4, 2, 9), ("bf16", 16, 336, 64, 6, 4, 3),
    ("bf16", 2, 33, 128, 5, 3, 2), ("fp32", 6, 77, 32, 9, 2, 5), ("fp32", 2, 16, 64, 1, 1, 0), ("fp32", 1, 1, 128, 3, 1, 2),
    ("fp32", 3, 65, 128, 3, 2, 1)])
def test_pages_of_the_caller(kind, heads, T, dh, n_kv, n_q, window):
    """The allocation-free call: pages and query tiles that 16, 32 and the key block do not divide, windows longer
    than the pages given.  fp32: sums of at most 700 products of order one, 1e-4 as in the other fp32 cases."""
    import torch
    from paper_2506_01380_b200 import nfd as N
    tdt = torch.bfloat16 if kind == "bf16" else torch.float32
    q, k, v = I.make_qkv(heads, dh, n_q * T, n_kv * T, seed=T + dh, bf16=kind == "bf16")
    tq, tk, tv = [torch.as_tensor(a).cuda().to(tdt) for a in (q, k, v)]
    pages = lambda x: x.view(heads, n_kv, T, dh).permute(1, 0, 2, 3).contiguous()
    out = torch.full((n_q * T, heads * dh), float("nan"), device="cuda", dtype=tdt)
    N.attention_noalloc(tq, pages(tk), pages(tv), n_q, window, out)
    got = out.float().cpu().numpy().astype(np.float64)
    ref = O.attention_block_causal(q, k, v, np.repeat(np.arange(n_kv - n_q, n_kv), T), np.repeat(np.arange(n_kv), T),
                                   window).transpose(1, 0, 2).reshape(n_q * T, heads * dh)
    tol = (TOL_ABS, TOL_REL) if kind == "bf16" else (1e-4, 1e-4)
    assert np.all(np.isfinite(got))
    assert np.abs(got - ref).max() <= tol[0] and np.linalg.norm(got - ref) / np.linalg.norm(ref) <= tol[1]
