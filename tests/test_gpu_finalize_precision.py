"""The sums of the chunk partials carry FP64's precision, however many chunks there are.

Members have disjoint cells, one per chunk, and values of 12 bits: every partial is exact in FP32
(a chunk's mass is the value, its product with the column sum the value's square), the sums over the
chunks need up to 53 bits, and FP64 holds them exactly in any order. IN_in is then one product and
one quotient of exact numbers, equal to the last bit."""
import numpy as np
import pytest

from tests.helpers import to_np

pytestmark = pytest.mark.gpu


# members, cells per chunk, and chunks (per SM: the streaming classes' groups; None: as many)
@pytest.mark.parametrize("mode", ["mean", "linear"])
@pytest.mark.parametrize("N,chunk,per_sm,chunks,scale", [
    (8, 128, 16, None, 8),        # one member per block of the finalisation
    (32, 128, 4, None, 9),
    (200, 256, 1, None, 10),      # 25 members per block
    (512, 512, 1, None, 10),
    (600, 8192, None, 64, 11),    # the member-blocked path
])
def test_exact_sums(mode, N, chunk, per_sm, chunks, scale):
    import torch
    from paper_2512_15187_gb300 import binding, build
    build.build()
    n = chunks or per_sm * torch.cuda.get_device_properties(0).multi_processor_count
    assert 24 + 2 * scale + np.ceil(np.log2(n)) <= 53
    rng = np.random.default_rng(N)
    k = rng.integers(2048, 4096, (N, n))
    v = k * 2.0 ** (-12 - rng.integers(0, scale + 1, (N, n)))
    U = torch.zeros((N, n * chunk), device="cuda")
    i = torch.arange(N, device="cuda")[:, None]
    U[i, torch.arange(n, device="cuda")[None, :] * chunk + i] = torch.from_numpy(v).float().cuda()
    h = binding.Handle(0)
    o = h.mean(U) if mode == "mean" else h.full(U, mode="linear")
    h.sync()
    want = (v * v).sum(axis=1) / (v.sum(axis=1) * N)
    np.testing.assert_array_equal(to_np(o["in_in"]), want)
    h.close()
