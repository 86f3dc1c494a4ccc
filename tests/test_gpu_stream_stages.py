"""The streaming pass of 257 to 512 members against the FP64 oracle where its 64-cell stages (up to
384 members) and whole-class boxes can go wrong: cell counts around one and two register tiles, chunks
that end in half a stage, member counts at the classes' edges, rows off the 16-byte boundary, and the
member maxima behind E4M3 scales.

Tolerance: the FP32 bar (1e-6) of every exact path, for which the order of the sums is unchanged."""
import numpy as np
import pytest

from oracle import pid_oracle as O
from paper_2512_15187_gb300 import synth
from tests.helpers import FP32_TOL, GRAM_TOL, assert_close, assert_rank_valid, to_np

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def H():
    from paper_2512_15187_gb300 import binding, build
    build.build()
    h = binding.Handle(0)
    yield h
    h.close()


def _dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


# 14592 = 152 x 96: chunks of three register tiles, one and a half stages each
@pytest.mark.parametrize("M", [1, 31, 32, 33, 64, 96, 100, 4863, 14592])
@pytest.mark.parametrize("N", [257, 320, 321, 384, 385, 448, 449, 512])
def test_stage_edges(H, N, M):
    U = synth.random_soft(N, M, seed=N + 7 * M, binary_frac=0.2)
    w = np.random.default_rng(M).uniform(0.2, 5, M).astype(np.float32) if (N + M) % 2 else None
    o = H.full(_dev(U), None if w is None else _dev(w), mode="linear")
    H.sync()
    for k, r in zip(("in_in", "in_out", "depth"), O.pid(U, w)):
        assert_close(to_np(o[k]), r, FP32_TOL, f"{N} x {M} {k}")
    assert_rank_valid(to_np(o["rank"]), to_np(o["depth"]))


@pytest.mark.parametrize("N", [260, 300, 384, 390])
@pytest.mark.parametrize("ld,shift", [(5003, 0), (5002, 0), (5004, 1), (5004, 2)])
def test_unaligned_rows_match_aligned_rows_bitwise(H, N, ld, shift):
    import torch
    M = 5001
    U = _dev(synth.random_soft(N, M, seed=N))
    rows = torch.zeros((N, 5004), device="cuda")
    rows[:, :M] = U
    buf = torch.full((N * ld + 8,), float("nan"), device="cuda")
    off = buf[shift:shift + N * ld].view(N, ld)[:, :M]
    off.copy_(U)
    a, b = H.full(rows[:, :M], mode="linear"), H.full(off, mode="linear")
    H.sync()
    for k in ("depth", "in_in", "in_out"):
        np.testing.assert_array_equal(to_np(a[k]), to_np(b[k]))


@pytest.mark.parametrize("N,M", [(300, 4097), (512, 4352)])
def test_maxima_give_the_scales(H, N, M):
    # members whose largest value spans many binades: a wrong maximum saturates or drowns E4M3
    U = synth.random_soft(N, M, seed=N) * (10.0 ** -np.linspace(0, 4, N)[:, None]).astype(np.float32)
    o = H.full(_dev(U), mode="full", precision="fp8")
    H.sync()
    assert_close(to_np(o["depth"]), O.pid(U)[2], GRAM_TOL, "E4M3 depth")
