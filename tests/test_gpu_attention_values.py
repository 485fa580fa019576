"""Attention on values that a fast softmax can get wrong: NaN in a key, at every place that a key can have among the
columns that one thread takes together; and how exact its probabilities are, for flat and for peaked rows."""
import pytest

from paper_2506_01380_b200 import inputs as I

pytestmark = pytest.mark.gpu


def _pages(heads, dh, T, n_kv, n_q, seed, dtype="bf16"):
    import torch
    tdt = torch.bfloat16 if dtype == "bf16" else torch.float32
    q, k, v = I.make_qkv(heads, dh, n_q * T, n_kv * T, seed=seed, bf16=dtype == "bf16")
    q, k, v = [torch.as_tensor(a).cuda().to(tdt) for a in (q, k, v)]
    pages = lambda x: x.view(heads, n_kv, T, dh).permute(1, 0, 2, 3).contiguous()
    return q, pages(k), pages(v), torch.empty(n_q * T, heads * dh, device="cuda", dtype=tdt)


@pytest.mark.parametrize("dtype,dh", [("bf16", 64), ("bf16", 32), ("bf16", 128), ("fp32", 64)])
def test_nan_in_a_key_reaches_every_row(dtype, dh):
    """A NaN score makes its row NaN, whichever key it belongs to: one key of 16 positions in turn, in the first and in
    the last block, for one head; the other heads stay finite."""
    import torch
    from paper_2506_01380_b200 import nfd as N
    heads, T, n_kv = 3, 336, 2
    q, k, v, out = _pages(heads, dh, T, n_kv, 1, seed=3, dtype=dtype)
    for page, key in [(0, i) for i in range(16)] + [(1, T - 1 - i) for i in range(16)]:
        kn = k.clone()
        kn[page, 1, key, 5] = float("nan")
        o = N.attention_noalloc(q, kn, v, 1, 1, out).view(T, heads, dh)
        assert torch.isnan(o[:, 1]).all(), (page, key)
        assert torch.isfinite(o[:, 0]).all() and torch.isfinite(o[:, 2]).all()


def _exact(q, k, v, n_q, window):
    """Softmax attention in 64 bits; q [H, n_q*T, dh], k and v [n_kv, H, T, dh]."""
    import torch
    n_kv, H, T, dh = k.shape
    out = torch.empty(n_q * T, H * dh, device="cuda", dtype=torch.float64)
    for j in range(n_q):
        f = n_kv - n_q + j
        kk, vv = [x[max(0, f - window):f + 1].double().permute(1, 0, 2, 3).reshape(H, -1, dh) for x in (k, v)]
        s = q[:, j * T:(j + 1) * T].double() @ kk.transpose(1, 2) / dh ** 0.5
        out[j * T:(j + 1) * T] = (torch.softmax(s, -1) @ vv).permute(1, 0, 2).reshape(T, H * dh)
    return out


def _rel(a, b):
    return float((a.double() - b).norm() / b.norm())


@pytest.mark.parametrize("scale", [1, 4])
@pytest.mark.parametrize("heads,dh,T,n_kv,n_q,window", [
    (16, 64, 336, 17, 1, 16), (12, 64, 220, 12, 2, 9), (4, 32, 64, 5, 1, 4), (4, 64, 128, 9, 4, 8), (8, 128, 100, 9, 2, 8)])
def test_bf16_result_is_as_exact_as_its_own_rounding(heads, dh, T, n_kv, n_q, window, scale):
    """The error against 64 bits is that of rounding the result to bf16 and no more: probabilities that lose 2^-17 add
    less than 1e-4 of it, probabilities rounded to bf16 (2^-9) add 40 %.  Both entry points."""
    import torch
    from paper_2506_01380_b200 import nfd as N
    q, k, v, out = _pages(heads, dh, T, n_kv, n_q, seed=T)
    q = q * scale
    ref = _exact(q, k, v, n_q, window)
    limit = 1.02 * _rel(ref.to(torch.bfloat16), ref)
    assert _rel(N.attention_noalloc(q, k, v, n_q, window, out), ref) <= limit
    if dh != 128:
        rope = dict(rope_t=16, rope_h=24, rope_w=24) if dh == 64 else dict(rope_t=8, rope_h=12, rope_w=12)
        cfg = I.make_cfg("nfd310m", n_layers=1, d_model=heads * dh, n_heads=heads, head_dim=dh, d_mlp=256, latent_h=T // 2,
                         latent_w=8, patch=2, ctx_frames=window, max_spec=4, **rope)
        assert I.tokens_per_frame(cfg) == T
        g = N.NFD(cfg, I.make_weights(cfg, 0))
        rows = lambda x: x.permute(1, 0, 2, 3).reshape(heads, n_kv * T, dh).contiguous()
        assert _rel(g.attention(q, rows(k), rows(v), n_q, n_kv, window), ref) <= limit
        assert g.status() == 0
