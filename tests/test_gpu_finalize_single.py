"""The Gram's finalisation on one CTA (up to 32 members with few chunks) and the cluster's just beyond
it, against the FP64 oracle: member counts around its limit and around a warp's rows, one chunk and
many, an empty member, tied members, batches that mix both.

Tolerance: split BF16 at 2e-5 (its products are exact to 2^-16); IN_in at the FP32 bar."""
import numpy as np
import pytest

from oracle import pid_oracle as O
from paper_2512_15187_gb300 import synth
from tests.helpers import FP32_TOL, assert_close, assert_rank_valid, to_np

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


def _masks(N, M):
    U = synth.random_soft(N, M, seed=N + M, binary_frac=0.2)
    if N > 3:
        U[1] = 0.0
        U[3] = U[0]
    return U


def _check(o, U):
    a, b, d = O.pid(U)
    assert_close(to_np(o["in_in"]), a, FP32_TOL, "in_in")
    assert_close(to_np(o["in_out"]), b, 2e-5, "in_out")
    assert_close(to_np(o["depth"]), d, 2e-5, "depth")
    assert_rank_valid(to_np(o["rank"]), to_np(o["depth"]))
    assert_close(to_np(o["P"]), O.inclusion_matrix(U), 2e-5, "P")


@pytest.mark.parametrize("N,M", [(1, 1), (2, 700), (15, 512), (16, 4096), (17, 30000), (31, 4096),
                                 (32, 16384), (32, 16896), (33, 4096)])
def test_parity(H, N, M):
    U = _masks(N, M)
    o = H.full(_dev(U), mode="full", precision="split_bf16", want_P=True)
    H.sync()
    _check(o, U)


def test_batches(H):
    shapes = [(5, 3000), (32, 4096), (20, 9001)]
    for more in ([], [(40, 5000)]):              # one CTA each, or clusters for all
        Us = [_masks(*s) for s in shapes + more]
        outs = H.batch([dict(data=_dev(U), mode="full", precision="split_bf16", want_P=True) for U in Us])
        H.sync()
        for o, U in zip(outs, Us):
            _check(o, U)
