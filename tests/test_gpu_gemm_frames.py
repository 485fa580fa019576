"""Projections of passes with many rows run in a kernel of their own, whose tiles may span frames, end inside a frame
and end inside the output columns: a batched pass has to equal single-frame passes bit for bit (every element's products
are summed in the same order in both kernels, and the single-frame path is compared with the oracle elsewhere)."""
import pytest

from paper_2506_01380_b200 import inputs as I

pytestmark = pytest.mark.gpu


# rows = streams * k * tokens; hidden 768 makes 18 column tiles of 128 for QKV, 6 for the residual projections
@pytest.mark.parametrize("hw,streams,k,act,dm,heads,fuse_ln", [
    ((48, 28), 1, 2, 0, 3072, 12, 1),       # 672 rows: one wave
    ((48, 28), 4, 2, 0, 3072, 12, 1),       # 2688 rows: several tiles per CTA, residual projections too
    ((48, 28), 4, 2, 1, 2730, 12, 1),       # gated, output columns that no tile divides
    ((48, 28), 4, 2, 0, 2052, 12, 0),       # stand-alone LayerNorm: plain bias
    ((48, 28), 3, 2, 0, 3072, 12, 1),       # 2016 rows: residual projections 96 wide, K split and not
    ((40, 22), 4, 3, 0, 3072, 12, 1),       # 220 tokens: frames end inside tiles and inside a warp's 32 rows
    ((16, 16), 8, 4, 1, 2048, 12, 1),       # 64 tokens: three frames in a tile
    ((46, 30), 4, 2, 0, 3072, 24, 1),       # 345 tokens, head dimension 32
    ((8, 6), 4, 4, 0, 4096, 12, 1),         # 12 tokens: eleven frames in a tile, more (u, v) pairs than epilogue threads
])
def test_batched_pass_equals_single_frames(hw, streams, k, act, dm, heads, fuse_ln):
    _batched_equals_single(768, hw, streams, k, act, dm, heads, fuse_ln)


@pytest.mark.parametrize("streams,k", [(5, 1), (3, 2)])
def test_tiles_of_three_groups_per_warp(streams, k):
    """1680 and 2016 rows onto 3072 columns: tiles 192 wide, of which a warp has three groups of 32, several tiles per CTA;
    warps whose rows belong to two frames store K and V themselves and Q through the two result boxes.  Repeated, for a
    store from a box that is overwritten too early is a matter of time."""
    _batched_equals_single(1024, (48, 28), streams, k, 0, 1024, 16, 1, passes=40)


@pytest.mark.parametrize("hw,act,dm,fuse_ln", [((48, 28), 0, 4096, 1), ((46, 30), 1, 2052, 1), ((48, 28), 0, 4100, 0)])
def test_mlp_of_a_single_frame_in_one_wave(hw, act, dm, fuse_ln):
    """4096 to 4104 columns: 43 tiles 96 wide, the last one 64 to 80, by three row blocks; the batched pass has wider ones."""
    _batched_equals_single(768, hw, 4, 2, act, dm, 12, fuse_ln)


def _batched_equals_single(d, hw, streams, k, act, dm, heads, fuse_ln, passes=1):
    import torch
    from paper_2506_01380_b200.nfd import NFD
    dh = d // heads
    rope = dict(rope_t=16, rope_h=24, rope_w=24) if dh == 64 else dict(rope_t=8, rope_h=12, rope_w=12)
    cfg = I.make_cfg("nfd310m", n_layers=2, d_model=d, n_heads=heads, head_dim=dh, d_mlp=dm, act=act, latent_h=hw[0],
                     latent_w=hw[1], ctx_frames=3, n_streams=streams, **rope)
    g = NFD(cfg, I.make_weights(cfg, 1, "stress"))
    g.set_option("fuse_ln", fuse_ln)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(hw[0])
    fs = I.frame_shape(cfg)
    x = torch.randn(streams, k, *fs, generator=gen, device="cuda")
    for s in range(streams):
        g.commit_frame(torch.randn(1 + s % 3, *fs, generator=gen, device="cuda"), [s] * (1 + s % 3), stream=s)
    acts = [(5 * s) % cfg["n_actions"] for s in range(streams)]
    one = torch.stack([torch.cat([g.denoise_step(x[s, j:j + 1].contiguous(), 0.6, acts[s], stream=s, offset=j) for j in range(k)])
                       for s in range(streams)])
    ref = [[g.kv_read(l, g.kv_state(s)[0] + j, stream=s) for l in (0, 1) for j in range(k)] for s in range(streams)]
    for _ in range(passes):
        both = g.denoise_step_batched(list(range(streams)), x, [0.6] * streams, acts)
        assert torch.isfinite(both).all() and torch.equal(both, one)
        for s in range(streams):
            new = [g.kv_read(l, g.kv_state(s)[0] + j, stream=s) for l in (0, 1) for j in range(k)]
            for a, b in zip(new, ref[s]):
                assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
    assert g.status() == 0
