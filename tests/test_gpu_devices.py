"""Contexts on several devices of one process."""
import pytest

from paper_2506_01380_b200 import inputs as I

pytestmark = pytest.mark.gpu


def test_a_context_on_every_device():
    """Kernel attributes (the shared memory a block may have) belong to a device: the second device's passes must run, on the
    same kernels, and give the first one's bits."""
    import torch
    from paper_2506_01380_b200.nfd import NFD
    if torch.cuda.device_count() < 2:
        pytest.skip("one device")
    cfg = I.make_cfg("nfd310m", n_layers=2, d_model=768, n_heads=12, d_mlp=3072, ctx_frames=2, n_streams=4)
    w = I.make_weights(cfg, 1)
    outs = []
    for dev in (0, 1):
        with torch.cuda.device(dev):
            g = NFD(cfg, w, device=f"cuda:{dev}")
            gen = torch.Generator(device="cpu")
            gen.manual_seed(1)
            x = torch.randn(4, 2, *I.frame_shape(cfg), generator=gen).cuda(dev)
            one = g.denoise_step(x[0], 0.6, 1)                                      # one tile per CTA, and attention
            many = g.denoise_step_batched([0, 1, 2, 3], x, [0.6] * 4, [1, 2, 3, 4])   # persistent tiles
            assert g.status() == 0
            outs.append((one.cpu(), many.cpu()))
    assert torch.equal(outs[0][0], outs[1][0]) and torch.equal(outs[0][1], outs[1][1])
