"""Which kernel a call runs, and whether it fills the SMs as its rule of dispatch says (launch records of the profiler)."""
import json

import pytest

from paper_2506_01380_b200 import inputs as I

pytestmark = [pytest.mark.gpu, pytest.mark.filterwarnings("ignore:.*Profiler clears events")]


def _events(call, tmp_path):
    import torch
    torch.cuda.synchronize()
    with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CPU, torch.profiler.ProfilerActivity.CUDA]) as p:
        call()
        torch.cuda.synchronize()
    p.export_chrome_trace(str(tmp_path / "t.json"))
    return json.load(open(tmp_path / "t.json"))["traceEvents"]


def _launches(call, tmp_path):
    """[(kernel name, registers per thread, CTAs, threads)] of the launches that `call` makes."""
    call()
    events = [e for e in _events(call, tmp_path) if e.get("cat") == "kernel"]
    if not events:
        pytest.skip("the profiler gives no launch records here")
    return [(e["name"], e["args"]["registers per thread"], e["args"]["grid"][0] * e["args"]["grid"][1] * e["args"]["grid"][2],
             e["args"]["block"][0]) for e in sorted(events, key=lambda e: e["ts"])]


def _pages(dtype, heads, dh, T, n_q, n_kv):
    import torch
    tdt = torch.bfloat16 if dtype == "bf16" else torch.float32
    zeros = lambda *s: torch.zeros(*s, device="cuda", dtype=tdt)
    return zeros(heads, n_q * T, dh), zeros(n_kv, heads, T, dh), zeros(n_q * T, heads * dh)


@pytest.mark.parametrize("dtype,heads,dh", [("fp32", 4, 32), ("bf16", 12, 32), ("bf16", 16, 64)])
def test_many_queries_on_the_fp32_pipes_leave_room_for_a_second_cta(dtype, heads, dh, tmp_path):
    """CTAs of 16 queries, 256 threads: two to an SM, 128 registers a thread, for head dimension 32 and for 64 in bf16 (the
    plain path of a bf16 context).  With one CTA to an SM these calls took up to a third longer."""
    from paper_2506_01380_b200 import nfd as N
    T, n_q = 336, 4
    if dtype == "fp32":
        q, k, out = _pages(dtype, heads, dh, T, n_q, 6)
        call = lambda: N.attention_noalloc(q, k, k, n_q, 2, out)
    else:
        rope = dict(rope_t=16, rope_h=24, rope_w=24) if dh == 64 else dict(rope_t=8, rope_h=12, rope_w=12)
        cfg = I.make_cfg("nfd310m", n_layers=1, d_model=heads * dh, n_heads=heads, head_dim=dh, d_mlp=256, ctx_frames=2, **rope)
        g = N.NFD(cfg, I.make_weights(cfg, 0))
        g.set_option("fast", 0)
        q, k, out = _pages(dtype, heads, dh, T, n_q, 6)
        rows = k.permute(1, 0, 2, 3).reshape(heads, 6 * T, dh).contiguous()
        call = lambda: g.attention(q, rows, rows, n_q, 6, 2, out=out)
    run = [x for x in _launches(call, tmp_path) if "k_attn_rows" in x[0]]
    assert len(run) == 1 and f"{dh}, 16, true>" in run[0][0] and run[0][2] == heads * n_q * T // 16 and run[0][3] == 256
    assert run[0][1] <= 128, run


@pytest.mark.parametrize("heads,T,n_q,instance", [
    (4, 40, 2, "8, false"), (4, 40, 8, "16, false"), (4, 77, 8, "16, true")])      # 24, 96 and 160 CTAs of 16 queries
def test_loads_in_flight_on_the_fp32_pipes_go_by_the_number_of_ctas(heads, T, n_q, instance, tmp_path):
    """Up to an SM's one CTA each, large batches of loads; beyond, small ones and room for a second."""
    from paper_2506_01380_b200 import nfd as N
    q, k, out = _pages("fp32", heads, 32, T, n_q, 9)
    run = [x for x in _launches(lambda: N.attention_noalloc(q, k, k, n_q, 2, out), tmp_path) if "k_attn_rows" in x[0]]
    assert len(run) == 1 and f"<float, 32, {instance}>" in run[0][0], run


@pytest.mark.parametrize("heads,dh,T,n_q,n_kv,window,kernel", [
    (16, 64, 336, 1, 17, 16, "k_attn_own"),       # 48 query tiles, 51 blocks: two pieces
    (16, 64, 336, 4, 12, 8, "k_attn_tc"),         # 192 query tiles: whole
    (4, 32, 77, 1, 5, 4, "k_attn_tc")])           # five blocks: a merge would take longer
def test_split_windows_of_the_caller_as_clusters_whole_ones_on_the_persistent_kernel(heads, dh, T, n_q, n_kv, window, kernel, tmp_path):
    from paper_2506_01380_b200 import nfd as N
    q, k, out = _pages("bf16", heads, dh, T, n_q, n_kv)
    run = _launches(lambda: N.attention_noalloc(q, k, k, n_q, window, out), tmp_path)
    assert len(run) == 2 and "k_set_params" in run[0][0] and kernel + "<" in run[1][0], run


def test_a_pass_has_one_graph_for_velocities_and_samplers(tmp_path):
    """The first velocity asked for behind a generation, and the first undistilled sample, replay the generation's graphs."""
    import torch
    from paper_2506_01380_b200 import nfd as N
    cfg = I.make_cfg("tiny_bf16")
    g = N.NFD(cfg, I.make_weights(cfg, 0))
    gen = torch.Generator(device="cuda")
    gen.manual_seed(1)
    noise = torch.randn(cfg["n_steps"], 1, *I.frame_shape(cfg), generator=gen, device="cuda")
    x, v = noise[0].contiguous(), torch.empty_like(noise[0])
    g.set_option("lazy_commit", 0)

    def made(call):
        return [e["name"] for e in _events(call, tmp_path) if "GraphInstantiate" in e.get("name", "")]

    if not made(lambda: g.speculate(1, 1, noise)):
        pytest.skip("the profiler gives no records of graphs here")
    g.rollback(1)
    g.speculate(1, 1, noise)                         # the modulation is cached now: graphs without conditioning
    g.rollback(1)
    for _ in range(2):                               # with conditioning and without
        assert not made(lambda: g.denoise_step(x, 0.77, 1, out=v))
    assert not made(lambda: g.sample_dpmpp(1, 1, x, n_evals=3))


@pytest.mark.parametrize("model", ["tiny_bf16", "tiny"])
def test_velocities_and_samples_in_turn(model):
    """The sampler's step is switched on and off in the one graph of a pass: a program that asks for velocities, generations and
    undistilled samples in turn gets what launches without graphs give."""
    import torch
    from paper_2506_01380_b200 import nfd as N
    cfg = I.make_cfg(model)
    w = I.make_weights(cfg, 3, "stress")
    gen = torch.Generator(device="cuda")
    gen.manual_seed(2)
    noise = [torch.randn(cfg["n_steps"], 2, *I.frame_shape(cfg), generator=gen, device="cuda") for _ in range(3)]
    outs = []
    for graph in (1, 0):
        g = N.NFD(cfg, w)
        g.set_option("graph", graph)
        out = []
        for i, n in enumerate(noise):
            out.append(g.denoise_step(n[0].contiguous(), 0.4 + 0.1 * i, 1))
            out.append(g.speculate(2, i, n))
            g.rollback(1)
            out.append(g.denoise_step(n[1].contiguous(), 0.9, 2))
            out.append(g.denoise_step(n[2].contiguous(), 0.9, 2))
            out.append(g.sample_dpmpp(2, i, n[0].contiguous(), n_evals=4))
            g.rollback(0)
        out.append(torch.tensor([g.kv_hash() % 2 ** 40], device="cuda"))
        assert g.status() == 0
        outs.append(out)
    for a, b in zip(*outs):
        assert torch.equal(a, b)
