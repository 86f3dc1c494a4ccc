"""GPU parity of the finalisation at the edges of its member blocks and dispatch rules: member
counts around the cluster's 8 blocks, the P launch above 96 members, Gram partials summed by
the finalisation itself or by a launch of their own, and sums that leave the FP32 range."""
import numpy as np
import pytest

from oracle import pid_oracle as O
from paper_2512_15187_gb300 import synth
from tests.helpers import (FP32_TOL, GRAM_TOL, assert_close, assert_rank_agrees_outside_ties,
                           assert_rank_valid, to_np)

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


def _check(o, ref, tol):
    for k, r in zip(("in_in", "in_out", "depth"), ref):
        assert_close(to_np(o[k]), r, FP32_TOL if k == "in_in" else tol, k)
    assert_rank_valid(to_np(o["rank"]), to_np(o["depth"]))
    assert_rank_agrees_outside_ties(to_np(o["rank"]), ref[2], tol)


# one to three members per CTA, the last CTAs empty or partly filled, 64 per CTA
@pytest.mark.parametrize("N", [1, 7, 8, 9, 17, 63, 65, 257, 511, 512])
@pytest.mark.parametrize("M", [128, 40000])     # one chunk, many chunks
def test_finalisation_member_blocks(H, N, M):
    U = synth.random_soft(N, M, seed=N + M, binary_frac=0.3)
    if N > 2:
        U[1] = U[0]                  # ties
        U[2] = 0.0                   # zero mass
    Ud = _dev(U)
    _check(H.mean(Ud), O.pid_mean(U), FP32_TOL)
    _check(H.full(Ud, mode="linear"), O.pid(U), FP32_TOL)
    r = np.random.default_rng(N).uniform(0.1, 2.0, N)
    _check(H.mean_weighted(Ud, _dev(r)), O.pid_mean_weighted(U, r), FP32_TOL)
    H.sync()


# P written by the finalisation (up to 96 members) and by its own launch; Gram partials of
# up to 2 MB summed inline (few chunks) or over the whole GPU (many)
@pytest.mark.parametrize("N,M", [(1, 300), (9, 4096), (96, 2048), (97, 2048), (97, 60000),
                                 (200, 1024), (257, 2000), (512, 5000)])
def test_gram_finalisation_paths(H, N, M):
    U = synth.random_soft(N, M, seed=3 * N + M, binary_frac=0.2)
    if N > 2:
        U[2] = 0.0
    o = H.full(_dev(U), mode="full", precision="split_bf16", want_P=True)
    H.sync()
    _check(o, O.pid(U), GRAM_TOL)
    assert_close(to_np(o["P"]), O.inclusion_matrix(U), GRAM_TOL, "P")
    assert 0.0 <= float(to_np(o["err_est"])[0]) <= 2e-5


def test_sums_beyond_the_fp32_range(H):
    """Chunk partials that are finite FP32 values but whose sum over the chunks is not."""
    U = synth.random_soft(4, 1 << 16, seed=8)
    w = np.full(U.shape[1], 1e35, dtype=np.float32)
    ref = O.pid_mean(U, w)
    assert O.mass(U, w).max() > 3.5e38
    o = H.mean(_dev(U), _dev(w))
    H.sync()
    _check(o, ref, FP32_TOL)


def test_nan_input_reaches_the_outputs(H):
    """One NaN cell (validation off): its member has no positive mass, every other member's
    product with the mean contour is NaN, and the mean contour has no positive mass."""
    U = synth.random_soft(20, 5000, seed=9)
    U[3, 77] = np.nan
    o = H.mean(_dev(U))
    H.sync()
    in_in = to_np(o["in_in"])
    assert in_in[3] == 0.0 and np.isnan(np.delete(in_in, 3)).all()
    assert (to_np(o["in_out"]) == 0.0).all() and (to_np(o["depth"]) == 0.0).all()
    assert to_np(o["rank"]).tolist() == list(range(20))


# beyond the cluster's 512 members: 32 members per CTA of the reduction, rank slices below,
# above and across the 1024 members of a block, one or several row groups of chunks
@pytest.mark.parametrize("N,M", [(513, 100), (545, 9001), (1023, 300), (1025, 70000), (2100, 1000)])
def test_large_ensemble_finalisation(H, N, M):
    U = synth.random_soft(N, M, seed=N + M, binary_frac=0.3)
    U[N - 1] = U[0]              # ties across the blocks
    U[N // 2] = U[0]
    U[5] = 0.0                   # zero mass
    Ud = _dev(U)
    _check(H.mean(Ud), O.pid_mean(U), FP32_TOL)
    _check(H.full(Ud, mode="linear"), O.pid(U), FP32_TOL)
    r = np.random.default_rng(N).uniform(0.1, 2.0, N)
    _check(H.mean_weighted(Ud, _dev(r)), O.pid_mean_weighted(U, r), FP32_TOL)
    H.sync()
