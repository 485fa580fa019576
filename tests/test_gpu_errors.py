"""Error paths of libnfd on the GPU, each made without a device fault: a launch that
the runtime refuses on the host, a pass descriptor with a bad index that the first
kernel of the pass catches, and a bounded device-side wait that runs out because the
producer left one pipeline stage out.  After each, the context must keep working and
give bitwise the results of a context that never saw the error."""
import numpy as np
import pytest

from paper_2506_01380_b200 import inputs as I

pytestmark = pytest.mark.gpu

E_CUDA, E_TIMEOUT, E_DEVICE = -7, -8, -9


def _pair(name="tiny_bf16", seed=13):
    import torch
    from paper_2506_01380_b200.nfd import NFD
    cfg = I.make_cfg(name)
    w = I.make_weights(cfg, seed, "stress")
    a, b = NFD(cfg, w), NFD(cfg, w)
    x0 = torch.as_tensor(I.make_latents(cfg, 2, 1)).cuda()
    for g in (a, b):
        g.commit_frame(x0, [1, 2])
    return cfg, a, b, torch


def _same_generation(cfg, a, b, torch, seed):
    noise = torch.as_tensor(I.make_noise(cfg, cfg["n_steps"], 2, seed)).cuda()
    ya, yb = a.speculate(2, 3, noise), b.speculate(2, 3, noise)
    assert torch.equal(ya, yb)
    a.rollback(1), b.rollback(1)
    assert a.kv_state() == b.kv_state() and a.kv_hash() == b.kv_hash()
    assert a.status() == 0 and b.status() == 0


@pytest.mark.parametrize("graph", [1, 0])
def test_refused_launch_fails_one_call_only(graph):
    from paper_2506_01380_b200.nfd import NfdError
    cfg, a, b, torch = _pair()
    a.set_option("graph", graph), b.set_option("graph", graph)
    noise = torch.as_tensor(I.make_noise(cfg, cfg["n_steps"], 2, 5)).cuda()
    s0 = a.kv_state()
    a.set_option("test_fail_launch", 1)
    with pytest.raises(NfdError) as e:
        a.speculate(2, 3, noise)
    assert e.value.code == E_CUDA
    assert a.kv_state() == s0, "a failed call must not count frames"
    assert a.status() == 0                       # a host-side refusal: nothing ran wrongly on the device
    _same_generation(cfg, a, b, torch, 6)        # the very next call works, and so do the ones after it
    _same_generation(cfg, a, b, torch, 7)


def test_bad_descriptor_is_caught_on_the_device():
    cfg, a, b, torch = _pair()
    x = torch.as_tensor(I.make_latents(cfg, 1, 3)).cuda()
    a.set_option("test_corrupt_desc", 1)
    a.denoise_step(x, 0.5, 1)                    # enqueued; the device finds the bad batch slot
    assert a.status() == E_DEVICE
    assert a.status() == E_DEVICE                # the latch keeps the code ...
    a.set_option("clear_status", 1)              # ... until it is cleared
    assert a.status() == 0
    # the redirected pass wrote into slot 0's pages: start both contexts afresh and compare
    x0 = torch.as_tensor(I.make_latents(cfg, 2, 1)).cuda()
    for g in (a, b):
        g.reset(0)
        g.commit_frame(x0, [1, 2])
    _same_generation(cfg, a, b, torch, 8)


@pytest.mark.parametrize("name", ["tiny_bf16", "nfd310m_slice"])
def test_expired_wait_surfaces_as_timeout_and_context_survives(name):
    """Every tensor-core GEMM's producer leaves out its last stage; the consumer's wait (limit shortened to
    200 microseconds) gives up, latches NFD_E_TIMEOUT and the kernel leaves by its normal exit."""
    cfg, a, b, torch = _pair(name)
    x = torch.as_tensor(I.make_latents(cfg, 1, 3)).cuda()
    a.set_option("test_wait_limit_us", 200)
    a.set_option("test_skip_stage", 1)
    a.denoise_step(x, 0.5, 1)
    assert a.status() == E_TIMEOUT
    a.set_option("test_skip_stage", 0)
    a.set_option("test_wait_limit_us", 0)
    a.set_option("clear_status", 1)
    assert a.status() == 0
    v1, v2 = a.denoise_step(x, 0.5, 1), b.denoise_step(x, 0.5, 1)
    assert torch.equal(v1, v2), "the context must compute as before once the switch is off"
    _same_generation(cfg, a, b, torch, 9)


def _late(g):
    g.set_option("test_wait_limit_us", 200)
    g.set_option("test_skip_stage", 1)


def _in_time(g):
    g.set_option("test_skip_stage", 0)
    g.set_option("test_wait_limit_us", 0)
    g.set_option("clear_status", 1)


def test_expired_wait_in_the_persistent_gemm():
    """A batched pass of 2688 rows: every projection, residual ones too, runs in the persistent kernel."""
    import torch
    from paper_2506_01380_b200.nfd import NFD
    cfg = I.make_cfg("nfd310m", n_layers=2, d_model=768, n_heads=12, d_mlp=3072, ctx_frames=2, n_streams=4)
    g = NFD(cfg, I.make_weights(cfg, 1, "stress"))
    gen = torch.Generator(device="cuda")
    gen.manual_seed(1)
    x = torch.randn(4, 2, *I.frame_shape(cfg), generator=gen, device="cuda")
    one = lambda: g.denoise_step_batched([0, 1, 2, 3], x, [0.6] * 4, [1, 2, 3, 4])
    ref = one()
    _late(g)
    one()
    assert g.status() == E_TIMEOUT
    _in_time(g)
    assert g.status() == 0
    assert torch.equal(one(), ref) and g.status() == 0


@pytest.mark.parametrize("streams,n_q", [(1, 1), (8, 4)])
def test_expired_wait_in_attention_leaves_nan(streams, n_q):
    """K does not come: the rows are NaN and not what the accumulators happened to hold, with split windows (whose counters
    must be at rest afterwards) and unsplit ones, several items per CTA."""
    import torch
    from paper_2506_01380_b200.nfd import NFD
    cfg = I.make_cfg("nfd310m", n_layers=1, ctx_frames=16, n_streams=streams)
    g = NFD(cfg, I.make_weights(cfg, 0))
    q, k, v = [torch.as_tensor(a).cuda().bfloat16() for a in I.make_qkv(16, 64, n_q * 336, 20 * 336, seed=5)]
    ref = g.attention(q, k, v, n_q, 20, 16)
    assert torch.isfinite(ref).all()
    _late(g)
    assert torch.isnan(g.attention(q, k, v, n_q, 20, 16)).all()
    assert g.status() == E_TIMEOUT
    _in_time(g)
    assert torch.equal(g.attention(q, k, v, n_q, 20, 16), ref) and g.status() == 0


def _caller_pages(heads, T, n_kv, seed=5):
    import torch
    q, k, v = [torch.as_tensor(a).cuda().bfloat16() for a in I.make_qkv(heads, 64, T, n_kv * T, seed=seed)]
    pages = lambda x: x.view(heads, n_kv, T, 64).permute(1, 0, 2, 3).contiguous()
    return q, pages(k), pages(v)


def _any_context():
    from paper_2506_01380_b200.nfd import NFD
    cfg = I.make_cfg("tiny_bf16")
    return NFD(cfg, I.make_weights(cfg, 0))


def test_refused_clusters_leave_the_windows_whole():
    """Where the runtime refuses the launch as clusters the call stays on the tensor cores, its windows whole: the bits of a
    call whose windows the plan leaves whole (78 query tiles), head by head, which neither the merge of two pieces nor the
    kernel on the fp32 pipes gives."""
    import torch
    from paper_2506_01380_b200 import nfd as N
    g, T, n_kv = _any_context(), 336, 17
    q, k, v = _caller_pages(26, T, n_kv)
    whole = N.attention_noalloc(q, k, v, 1, 16, torch.empty(T, 26 * 64, device="cuda", dtype=torch.bfloat16))
    q, k, v = q[:16].contiguous(), k[:, :16].contiguous(), v[:, :16].contiguous()
    call = lambda: N.attention_noalloc(q, k, v, 1, 16, torch.full((T, 16 * 64), float("nan"), device="cuda", dtype=torch.bfloat16))
    split = call()
    g.set_option("test_noalloc", 2)
    refused = call()
    assert torch.equal(refused, whole[:, :16 * 64]) and not torch.equal(refused, split)
    assert torch.equal(call(), split)                # one call only


@pytest.mark.parametrize("heads,T", [(16, 336), (1, 336), (3, 100), (26, 336)])    # 2, 8 and 6 pieces, whole windows
def test_expired_wait_in_the_allocation_free_call_leaves_nan(heads, T):
    """K does not come: every wait behind it gives up (after 0.4 s), the rows are NaN, the CTAs of the clusters all leave, and
    the next call computes as ever."""
    import torch
    from paper_2506_01380_b200 import nfd as N
    g = _any_context()
    q, k, v = _caller_pages(heads, T, 17)
    call = lambda: N.attention_noalloc(q, k, v, 1, 16, torch.zeros(T, heads * 64, device="cuda", dtype=torch.bfloat16))
    ref = call()
    assert torch.isfinite(ref).all()
    g.set_option("test_noalloc", 1)
    assert torch.isnan(call()).all()
    assert torch.equal(call(), ref)
