"""Launches of the two attention entry points, captured: the attention kernel reads its descriptor at once, so the kernel
that writes the descriptor has to end before it starts.  A programmatic edge would let it start earlier."""
import ctypes as C

import pytest

from paper_2506_01380_b200 import inputs as I

pytestmark = pytest.mark.gpu

THREAD_LOCAL, DEFAULT_EDGE = 1, 0


def _edge_types(stream, call):
    """Types of the edges of the graph that `call` is captured as (cuGraphGetEdges_v2: 8 bytes per edge, the third is it)."""
    drv = C.CDLL("libcuda.so.1")
    h, graph = C.c_void_p(stream.cuda_stream), C.c_void_p()
    assert drv.cuStreamBeginCapture_v2(h, THREAD_LOCAL) == 0
    try:
        call()
    finally:
        rc = drv.cuStreamEndCapture(h, C.byref(graph))
    assert rc == 0
    n = C.c_size_t(0)
    assert drv.cuGraphGetEdges_v2(graph, None, None, None, C.byref(n)) == 0
    a, b, data = (C.c_void_p * n.value)(), (C.c_void_p * n.value)(), (C.c_ubyte * (8 * n.value))()
    assert drv.cuGraphGetEdges_v2(graph, a, b, data, C.byref(n)) == 0
    assert drv.cuGraphDestroy(graph) == 0
    return [data[8 * i + 2] for i in range(n.value)]


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
def test_allocation_free_attention_in_plain_order(dtype):
    import torch
    from paper_2506_01380_b200 import nfd as N
    tdt = torch.bfloat16 if dtype == "bf16" else torch.float32
    H, T, dh = 4, 80, 64
    q, out = torch.zeros(H, T, dh, device="cuda", dtype=tdt), torch.zeros(T, H * dh, device="cuda", dtype=tdt)
    k = torch.zeros(3, H, T, dh, device="cuda", dtype=tdt)
    st = torch.cuda.Stream()
    st.wait_stream(torch.cuda.current_stream())
    call = lambda: N.attention_noalloc(q, k, k, 1, 2, out, stream=st)
    call()                                   # symbol look-up
    torch.cuda.synchronize()
    types = _edge_types(st, call)
    assert len(types) == 1 and types == [DEFAULT_EDGE]


def test_context_attention_in_plain_order():
    import torch
    from paper_2506_01380_b200 import nfd as N
    cfg = I.make_cfg("nfd310m", n_layers=1, ctx_frames=2)
    g = N.NFD(cfg, I.make_weights(cfg, 0))
    H, T = cfg["n_heads"], I.tokens_per_frame(cfg)
    q, k = [torch.zeros(H, n * T, 64, device="cuda", dtype=torch.bfloat16) for n in (1, 3)]
    out = g.attention(q, k, k, 1, 3, 2)
    torch.cuda.synchronize()
    with torch.cuda.stream(g.stream):
        types = _edge_types(g.stream, lambda: g.attention(q, None, None, 1, 3, 2, out=out))
    assert len(types) == 3 and types == [DEFAULT_EDGE] * 3      # copy -> descriptor -> attention -> copy
