"""How the attention kernels' work is cut into items (csrc/nfd_attn_plan.h), on the CPU: the plan of a configuration."""
import ctypes as C
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = r"""
#include "nfd_attn_plan.h"
extern "C" void own_plan(int T, int tiles, int n_blocks, const int *clusters, int *out) {
    AttnPlan pl;
    attn_blocks(pl, T);
    attn_own_plan(pl, tiles, n_blocks, [&](int k) { return clusters[k]; });
    out[0] = pl.MAXSPLIT, out[1] = pl.CH;
}
// The plan of a configuration.
extern "C" int context_plan(int T, int heads, int n_streams, int window, int n_sm, int *out) {
    AttnPlan pl;
    attn_blocks(pl, T);
    const int n_blocks = (window + 1) * pl.BPF;
    attn_split_plan(pl, heads * pl.QT, n_streams, n_blocks, n_sm);
    if (!attn_divisors(pl, 32, window, n_sm)) return 0;
    out[0] = pl.WH, out[1] = pl.SP, out[2] = pl.MAXSPLIT, out[3] = pl.CH, out[4] = n_blocks, out[5] = pl.BPF, out[6] = pl.QT;
    return 1;
}
// Every item of a pass of `frames` frames, whose windows are full: seen[(frame, tile) * MAXSPLIT + split] counts it, load[c] is
// the time of CTA c in half blocks (a whole item a block more than it has, a piece two and a half), turn[c] the same where the pieces
// follow the whole items in turn; the largest number of items of a CTA, -1 where an item is out of range.
extern "C" int deal(int T, int heads, int n_streams, int window, int n_sm, int frames, int *seen, int *load, int *turn) {
    AttnPlan pl;
    attn_blocks(pl, T);
    const int n_blocks = (window + 1) * pl.BPF, tiles = heads * pl.QT;
    attn_split_plan(pl, tiles, n_streams, n_blocks, n_sm);
    if (!attn_divisors(pl, 32, window, n_sm)) return -2;
    attn_deal(pl, frames, n_sm);
    int items = 0;
    for (int c = 0; c < pl.grid; ++c) {
        const int n = pl.dealt() ? attn_dealt_count(c, pl) : (pl.n_items - c + pl.grid - 1) / pl.grid;
        for (int i = 0; i < n; ++i) {
            const int item = pl.dealt() ? attn_dealt(c, i, pl) : c + i * pl.grid;
            if (item < 0 || item >= pl.n_items) return -1;
            const AttnPlace p = pl.dealt() ? attn_place<true>(item, pl) : attn_place<false>(item, pl);
            if (p.j < 0 || p.j >= frames || p.t < 0 || p.t >= tiles || p.split < 0 || p.split >= pl.MAXSPLIT) return -1;
            if (p.whole != (p.t < pl.WH) || (!p.whole && p.tile != p.j * pl.SP + p.t - pl.WH)) return -1;
            ++seen[(p.j * tiles + p.t) * pl.MAXSPLIT + p.split];
            load[c] += p.whole || pl.MAXSPLIT == 1 ? 2 * (n_blocks + 1) : 2 * pl.CH + 5;
        }
        if (n > items) items = n;
        if (n < 1) return -1;
    }
    for (int i = 0; i < pl.n_items; ++i)
        turn[i % pl.grid] += i < pl.whole || pl.MAXSPLIT == 1 ? 2 * (n_blocks + 1) : 2 * pl.CH + 5;
    return items;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    (d / "plan.cpp").write_text(SOURCE)
    subprocess.run([shutil.which("g++") or "g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_2506_01380_b200", "csrc"), "-o", str(d / "plan.so"), str(d / "plan.cpp")], check=True)
    return C.CDLL(str(d / "plan.so"))


# clusters of k CTAs that a 148-SM B200 holds at once, k = 0 .. 8
B200 = [0, 148, 74, 45, 33, 26, 22, 15, 15]


@pytest.mark.parametrize("T", [40, 77, 220, 336])
def test_clusters_of_the_caller_s_pages_fit_the_machine(lib, T):
    """Every tile's cluster is resident at once, on a whole B200, and on a machine that holds few or no clusters."""
    out = (C.c_int * 2)()
    for machine in (B200, [0, 148, 74, 45, 33, 0, 0, 0, 0], [0, 20, 10, 4, 2, 1, 1, 1, 1], [0, 20] + [0] * 7):
        for tiles in range(1, 160):
            for n_blocks in (1, 2, 9, 33, 51, 400):
                lib.own_plan(T, tiles, n_blocks, (C.c_int * 9)(*machine), out)
                k, ch = out
                assert k == 1 or tiles <= machine[k], (machine, tiles, n_blocks, k)
                assert 1 <= k <= n_blocks and (k - 1) * ch < n_blocks <= k * ch
    # windows that are too short for a merge stay whole: 6 blocks of 96 keys, 8 and 9 of 64; not 8 and 10
    for tokens, n_blocks, split in ((96, 6, False), (40, 8, False), (40, 9, False), (96, 8, True), (40, 10, True)):
        lib.own_plan(tokens, 8, n_blocks, (C.c_int * 9)(*B200), out)
        assert (out[0] > 1) == split, (tokens, n_blocks)
    lib.own_plan(40, 16, 33, (C.c_int * 9)(*B200), out)
    assert out[0] not in (7, 8)          # 16 clusters of either do not fit


SHAPES = [(336, 16, 32), (336, 16, 16), (336, 24, 16), (336, 12, 16), (220, 12, 9), (220, 16, 16), (390, 24, 8), (64, 4, 32),
          (96, 24, 8), (336, 3, 31)]                        # tokens, heads, window


@pytest.mark.parametrize("T,heads,window", SHAPES)
def test_every_item_is_dealt_out_once_and_no_cta_is_busier_than_in_turn(lib, T, heads, window):
    """Passes of 1 to 32 frames in contexts of 1 to 9 streams: every piece of every query tile comes up once, and the busiest CTA of
    a pass of no more frames than streams has no more to do than with the pieces dealt on in turn behind the whole items, half a
    piece aside."""
    info = (C.c_int * 7)()
    for n_sm in (148, 132, 20):
        for streams in range(1, 10):
            assert lib.context_plan(T, heads, streams, window, n_sm, info)
            wh, sp, k, ch, n_blocks, bpf, qt = info
            tiles = heads * qt
            assert wh + sp == tiles and (k - 1) * ch < n_blocks <= k * ch
            for frames in sorted({1, 2, 3, 4, 5, 6, 7, 8, streams, 2 * streams, 16, 31, 32}):
                seen, load, turn = (C.c_int * (frames * tiles * k))(), (C.c_int * n_sm)(), (C.c_int * n_sm)()
                items = lib.deal(T, heads, streams, window, n_sm, frames, seen, load, turn)
                assert 0 < items <= 2048
                want = [1 if t >= wh or s == 0 else 0 for _ in range(frames) for t in range(tiles) for s in range(k)]
                assert list(seen) == want, (n_sm, streams, frames)
                assert sum(load) == sum(turn)
                if frames <= streams:
                    assert max(load) <= max(turn) + ch, (n_sm, streams, frames)


def _start_plan(tiles, streams, n_blocks, n_sm):
    """The split of several streams as it was chosen at first, from its definition: (whole pairs, blocks of a piece)."""
    best = None
    for k in range(1, min(8, n_blocks) + 1):
        ch = -(-n_blocks // k)
        split = -(-n_blocks // ch)
        for wh in [tiles] if k == 1 else range(tiles):
            nw = streams * wh
            n = nw + streams * (tiles - wh) * split
            grid = min(n, n_sm)
            most = max(w * (n_blocks + 1) + (n // grid + (c < n % grid) - w) * (ch + 2.5)
                       for c in (0, nw % grid, n % grid) for w in [nw // grid + (c < nw % grid)])
            if best is None or most < best[0]:
                best = (most, 0 if k == 1 else wh, ch)
    return best[1:]


@pytest.mark.parametrize("T,heads,window", SHAPES)
def test_order_of_the_sums_of_several_streams(lib, T, heads, window):
    """The plan decides in which order a frame's sums are taken: windows of up to 33 frames keep the one they have."""
    info = (C.c_int * 7)()
    for streams in range(2, 10):
        assert lib.context_plan(T, heads, streams, window, 148, info)
        assert (info[0], info[3]) == _start_plan(heads * info[6], streams, info[4], 148)


@pytest.mark.parametrize("T,heads,streams,window", [(64, 4, 2, 1000), (128, 2, 3, 400), (64, 4, 4, 200), (64, 4, 1, 1000)])
def test_long_windows_of_few_heads_fill_the_machine(lib, T, heads, streams, window):
    """With a few query tiles to a frame and hundreds of blocks to a window the pieces of a frame of every stream fill more than
    half of the SMs.  (At most eight pieces a tile: 64 to 128 CTAs, windows up to 2.2 times as long.)"""
    info = (C.c_int * 7)()
    assert lib.context_plan(T, heads, streams, window, 148, info)
    assert 74 < info[1] * info[2] * streams <= 148 and info[0] == 0


def test_configuration_whose_pieces_are_counted_in_two_sweeps(lib):
    """32 heads, 336 tokens, four streams behind 12 frames, 32 frames in a pass: some CTA has more than the 32 items that one sweep of
    a warp counts (its values are checked on the GPU)."""
    frames, info = 32, (C.c_int * 7)()
    assert lib.context_plan(336, 32, 4, 12, 148, info) and info[2] > 1
    seen, load, turn = (C.c_int * (frames * 96 * info[2]))(), (C.c_int * 148)(), (C.c_int * 148)()
    assert lib.deal(336, 32, 4, 12, 148, frames, seen, load, turn) > 32


@pytest.mark.parametrize("heads,taken", [(9398, True), (9472, True), (9473, False)])
def test_items_of_one_kind_fill_a_cta_s_account(lib, heads, taken):
    """32 frames x heads x one query tile, whole windows: 2048 items to each of 148 CTAs are taken."""
    assert lib.context_plan(128, heads, 1, 1, 148, (C.c_int * 7)()) == taken
