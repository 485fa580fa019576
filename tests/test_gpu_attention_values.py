"""Attention on values that a fast softmax can get wrong: NaN in a key, at every place that a key can have among the
columns that one thread takes together."""
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
