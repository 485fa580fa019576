"""Attention on values that a fast softmax can get wrong: NaN in a key, at every place that a key can have among the
columns that one thread takes together; how exact its probabilities are, for flat and for peaked rows; scores that rise
beyond what the first ones are a reference for, scores of -inf, and pages smaller than a tile of keys."""
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


@pytest.mark.parametrize("streams,heads,T,window,n_kv,n_q", [
    (4, 16, 336, 16, 17, 8),         # 33 of 48 (head, query tile) pairs whole, 15 in three pieces
    (8, 16, 336, 32, 20, 3),         # 33 whole, 15 in three pieces of which the window fills two
    (3, 12, 220, 9, 12, 2),          # all in two pieces
    (2, 4, 64, 16, 17, 8)])          # all in six pieces, the last one shorter
def test_windows_whole_and_in_pieces(streams, heads, T, window, n_kv, n_q):
    """Contexts of several streams split the key ranges of some (head, query tile) pairs and not those of others."""
    from paper_2506_01380_b200 import nfd as N
    q, k, v, _ = _pages(heads, 64, T, n_kv, n_q, seed=T + streams)
    ref = _exact(q, k, v, n_q, window)
    cfg = I.make_cfg("nfd310m", n_layers=1, d_model=heads * 64, n_heads=heads, head_dim=64, d_mlp=256, latent_h=T // 2,
                     latent_w=8, patch=2, ctx_frames=window, max_spec=8, n_streams=streams)
    g = N.NFD(cfg, I.make_weights(cfg, 0))
    rows = lambda x: x.permute(1, 0, 2, 3).reshape(heads, n_kv * T, 64).contiguous()
    for _ in range(2):               # (the counters of the pieces are at rest after a call)
        assert _rel(g.attention(q, rows(k), rows(v), n_q, n_kv, window), ref) <= 1.02 * _rel(ref.bfloat16(), ref)
    assert g.status() == 0


def _rising(heads, dh, T, n_kv, n_q, seed, nats, v_scale=1.0):
    """Scores that rise by `nats` from the first page to the last, evenly: q has 8 in one column, and k there what it takes.
    The first rows of q take no part in it."""
    import torch
    q, k, v, out = _pages(heads, dh, T, n_kv, n_q, seed)
    q[:, :, 3] = 8
    q[:, :5, 3] = 0
    k[..., 3] = (torch.arange(n_kv, device="cuda") * (nats * dh ** 0.5 / 8 / max(n_kv - 1, 1))).view(n_kv, 1, 1).to(k.dtype)
    return q, k, v * v_scale, out


# Every item is walked again (the rise passes 2^100 over the item's first scores); a bf16 result within its own rounding.
@pytest.mark.parametrize("heads,T,streams,n_kv,n_q,window", [
    (16, 336, 8, 33, 8, 32),         # unsplit long windows, several items per CTA
    (16, 336, 1, 17, 1, 16),         # split windows
    (16, 220, 1, 17, 4, 16),         # pages that no block divides, several items per CTA
    (2, 64, 1, 40, 2, 39),           # one block per page
])
def test_scores_that_rise_beyond_the_reference(heads, T, streams, n_kv, n_q, window):
    import torch
    from paper_2506_01380_b200 import nfd as N
    q, k, v, out = _rising(heads, 64, T, n_kv, n_q, seed=T, nats=40 * n_kv)
    ref = _exact(q, k, v, n_q, window)
    limit = 1.02 * _rel(ref.to(torch.bfloat16), ref)
    cfg = I.make_cfg("nfd310m", n_layers=1, d_model=heads * 64, n_heads=heads, d_mlp=256, latent_h=T // 2, latent_w=8,
                     ctx_frames=window, max_spec=8, n_streams=streams)
    g = N.NFD(cfg, I.make_weights(cfg, 0))
    rows = lambda x: x.permute(1, 0, 2, 3).reshape(heads, n_kv * T, 64).contiguous()
    one = g.attention(q, rows(k), rows(v), n_q, n_kv, window)
    assert _rel(one, ref) <= limit
    assert torch.equal(one, g.attention(q, None, None, n_q, n_kv, window))
    # a frame alone and with others
    last = g.attention(q[:, -T:].contiguous(), None, None, 1, n_kv, window)
    assert torch.equal(last, one[-T:])
    assert g.status() == 0
    assert _rel(N.attention_noalloc(q, k, v, n_q, window, out), ref) <= limit


@pytest.mark.parametrize("heads,n_kv", [
    (2, 1201),          # 6 query tiles: eight pieces each, 451 blocks and fewer to a CTA
    (26, 301)])         # 78, more than clusters of two fit: one CTA to a tile, 903 blocks
def test_rising_scores_over_a_long_window(heads, n_kv):
    """The same with hundreds of frames in the window of the allocation-free call, in pieces and whole."""
    import torch
    from paper_2506_01380_b200 import nfd as N
    T = 336
    q, k, v, out = _rising(heads, 64, T, n_kv, 1, seed=1, nats=400)
    got = N.attention_noalloc(q, k, v, 1, n_kv, out)
    ref = torch.cat([_exact(q[h:h + 1], k[:, h:h + 1], v[:, h:h + 1], 1, n_kv) for h in range(heads)], dim=1)
    assert _rel(got, ref) <= 1.02 * _rel(ref.to(torch.bfloat16), ref)


def test_sums_that_leave_fp32_before_the_guard_of_the_scores():
    """Scores rise by 60 nats only, but with values of 2^80 the unnormalised sums pass 2^127."""
    import torch
    from paper_2506_01380_b200 import nfd as N
    q, k, v, out = _rising(4, 64, 220, 12, 2, seed=2, nats=60, v_scale=2.0 ** 80)
    got = N.attention_noalloc(q, k, v, 2, 11, out)
    ref = _exact(q, k, v, 2, 11)
    assert _rel(got, ref) <= 1.02 * _rel(ref.to(torch.bfloat16), ref)


@pytest.mark.parametrize("pages", [0, 3])
def test_scores_of_minus_infinity_count_for_nothing(pages):
    """The first 16 keys, or all keys of the first pages (more than a split takes), at -inf."""
    import torch
    from paper_2506_01380_b200 import nfd as N
    heads, T, n_kv, window = 16, 336, 17, 16
    q, k, v, out = _pages(heads, 64, T, n_kv, 1, seed=9)
    q[:, :, 0] = 1
    if pages:
        k[:pages, :, :, 0] = float("-inf")
    else:
        k[0, :, :16, 0] = float("-inf")
    ref = _exact(q, k, v, 1, window)
    limit = 1.02 * _rel(ref.to(torch.bfloat16), ref)
    cfg = I.make_cfg("nfd310m", n_layers=1, ctx_frames=window)
    g = N.NFD(cfg, I.make_weights(cfg, 0))
    rows = lambda x: x.permute(1, 0, 2, 3).reshape(heads, n_kv * T, 64).contiguous()
    assert _rel(g.attention(q, rows(k), rows(v), 1, n_kv, window), ref) <= limit
    assert _rel(N.attention_noalloc(q, k, v, 1, window, out), ref) <= limit


@pytest.mark.parametrize("dtype,dh,tol", [("fp32", 64, 1e-5), ("bf16", 128, 4e-3)])
def test_tiles_of_minus_infinity_on_the_fp32_pipes(dtype, dh, tol):
    """A warp's whole first tile of 32 keys at -inf, with finite ones after it.  fp32: sums of some hundred products of order
    one; bf16: half a unit in the last place of the result."""
    import torch
    from paper_2506_01380_b200 import nfd as N
    T, n_kv = 336, 3
    q, k, v, out = _pages(4, dh, T, n_kv, 1, seed=4, dtype=dtype)
    q[:, :, 0] = 1
    k[0, :, 64:130, 0] = float("-inf")
    k[0, :, 200:270, 0] = float("-inf")
    assert _rel(N.attention_noalloc(q, k, v, 1, 2, out), _exact(q, k, v, 1, 2)) <= tol


@pytest.mark.parametrize("T", [1, 2, 3, 5, 15, 16, 17, 31, 32, 33])
@pytest.mark.parametrize("dtype,dh,tol", [("fp32", 64, 1e-5), ("bf16", 128, 4e-3)])
def test_small_pages_on_the_fp32_pipes(T, dtype, dh, tol):
    """Several pages to a tile of 32 keys, the last tile with fewer; the tolerances of the case above."""
    from paper_2506_01380_b200 import nfd as N
    q, k, v, out = _pages(3, dh, T, 37, 2, seed=T, dtype=dtype)
    for window in (36, 5, 0):
        assert _rel(N.attention_noalloc(q, k, v, 2, window, out), _exact(q, k, v, 2, window)) <= tol


@pytest.mark.parametrize("nats", [0, 30])          # (30 nats a page: items are walked again)
@pytest.mark.parametrize("heads,T,dh,n_kv,n_q,window", [
    (16, 336, 64, 17, 1, 16),        # two pieces of 26 and 25 blocks
    (2, 100, 32, 9, 3, 8),           # pages of one masked block, head dimension 32
    (2, 64, 64, 8, 8, 8),            # windows of one to eight blocks: some have fewer pieces than the cluster has CTAs
    (1, 336, 64, 17, 1, 16)])        # eight pieces, the last one shorter
def test_pieces_as_the_ctas_of_a_cluster(heads, T, dh, n_kv, n_q, window, nats):
    import torch
    from paper_2506_01380_b200 import nfd as N
    q, k, v, out = _rising(heads, dh, T, n_kv, n_q, seed=T, nats=nats * n_kv) if nats else _pages(heads, dh, T, n_kv, n_q, seed=T)
    ref = _exact(q, k, v, n_q, window)
    got = N.attention_noalloc(q, k, v, n_q, window, out.fill_(float("nan")))
    assert _rel(got, ref) <= 1.02 * _rel(ref.to(torch.bfloat16), ref)


@pytest.mark.parametrize("streams,heads,hw,window,used,k", [
    (8, 16, (48, 28), 32, (2, 5), 1),        # 37 of 48 (head, query tile) pairs whole: batches that leave CTAs without a whole window
    (5, 16, (48, 28), 16, (3, 5), 2),        # 28 of 48, two frames a stream
    (4, 12, (40, 22), 9, (4,), 8),           # every pair in three pieces: 72 items a frame, 32 frames
    (4, 32, (48, 28), 12, (4,), 8)])         # 70 of 96, 32 frames: more than 32 items to a CTA, counted in two sweeps
def test_a_frame_s_bits_do_not_depend_on_the_batch(streams, heads, hw, window, used, k):
    """Contexts of several streams deal whole windows and pieces out to the CTAs by the number of frames in the pass; a frame's
    bits are those that it has alone."""
    import torch
    from paper_2506_01380_b200 import nfd as N
    cfg = I.make_cfg("nfd310m", n_layers=1, d_model=heads * 64, n_heads=heads, d_mlp=256, latent_h=hw[0], latent_w=hw[1],
                     ctx_frames=window, max_spec=8, n_streams=streams)
    g = N.NFD(cfg, I.make_weights(cfg, 0, "stress"))
    gen = torch.Generator(device="cuda")
    gen.manual_seed(window)
    fs = I.frame_shape(cfg)
    for s in range(streams):
        for n in range(0, window - s, 8):            # (windows of different lengths)
            m = min(8, window - s - n)
            g.commit_frame(torch.randn(m, *fs, generator=gen, device="cuda"), [1] * m, stream=s)
    x = torch.randn(streams, k, *fs, generator=gen, device="cuda")
    one = [torch.cat([g.denoise_step(x[s, j:j + 1].contiguous(), 0.6, s, stream=s, offset=j) for j in range(k)]) for s in range(max(used))]
    for n in used:
        for _ in range(2):
            both = g.denoise_step_batched(list(range(n)), x[:n].contiguous(), [0.6] * n, list(range(n)))
            assert torch.isfinite(both).all() and torch.equal(both, torch.stack(one[:n]))
    assert g.status() == 0


@pytest.mark.parametrize("T", [5, 33, 77])
@pytest.mark.parametrize("dtype,dh,tol", [("fp32", 32, 1e-5), ("fp32", 64, 1e-5), ("fp32", 128, 1e-5), ("bf16", 128, 4e-3)])
def test_sixteen_queries_to_a_cta_on_the_fp32_pipes(T, dtype, dh, tol):
    """With 60 heads CTAs take 16 queries (a last one with fewer), with 3 of them 8: a row's bits are the same.  Pages of 5 tokens
    are several to a tile.  The tolerances of the small pages above."""
    import torch
    from paper_2506_01380_b200 import nfd as N
    n_kv, n_q = 11, 2
    q, k, v, out = _pages(60, dh, T, n_kv, n_q, seed=T + dh, dtype=dtype)
    few = torch.empty(n_q * T, 3 * dh, device="cuda", dtype=out.dtype)
    for window in (10, 3):
        N.attention_noalloc(q, k, v, n_q, window, out)
        assert _rel(out, _exact(q, k, v, n_q, window)) <= tol
        N.attention_noalloc(q[:3].contiguous(), k[:, :3].contiguous(), v[:, :3].contiguous(), n_q, window, few)
        assert torch.equal(few, out[:, :3 * dh])
