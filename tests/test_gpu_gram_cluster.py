"""The one-pass cluster Gram (256 < N <= 512 members with enough cell chunks) against the FP64 oracle
and against the same cells as a short ensemble's tiles: ragged member blocks, cell counts that leave
the last stage, the last chunk and a cluster's share uneven, rows off the 16-byte boundary, fields.

Tolerances: the Gram bar for depths and P, the FP32 bar for IN_in; and a raw (pre-calibration) error
of 2e-5 for split BF16, whose products are exact to 2^-16 and summed in FP32."""
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


def _check(o, U, w, what):
    a, b, d = O.pid(U, w)
    assert_close(to_np(o["in_in"]), a, FP32_TOL, what + " in_in")
    assert_close(to_np(o["in_out"]), b, GRAM_TOL, what + " in_out")
    assert_close(to_np(o["depth"]), d, GRAM_TOL, what + " depth")
    assert_rank_valid(to_np(o["rank"]), to_np(o["depth"]))
    if "P" in o:
        assert_close(to_np(o["P"]), O.inclusion_matrix(U, w), GRAM_TOL, what + " P")


# 28 chunks of 4096 cells on 28 clusters, 33 and 60 chunks that clusters share
@pytest.mark.parametrize("prec", ["bf16", "split_bf16", "fp8"])
@pytest.mark.parametrize("N,M,weighted", [(257, 114688, False), (384, 135169, True), (391, 114689, True),
                                          (512, 245760, False)])
def test_parity(H, prec, N, M, weighted):
    U = synth.random_soft(N, M, seed=N + M, binary_frac=0.2)
    w = np.random.default_rng(M).uniform(0.2, 5, M).astype(np.float32) if weighted else None
    o = H.full(_dev(U), None if w is None else _dev(w), mode="full", precision=prec,
               want_P=prec != "fp8", want_err=True)
    H.sync()
    _check(o, U, w, f"{prec} {N} x {M}")
    if prec == "split_bf16":
        assert float(to_np(o["err_est"])[0]) <= 2e-5


@pytest.mark.parametrize("shift", [0, 1])
def test_binary_masks_row_offsets(H, shift):
    # 0/1 masks: every product and sum is a whole number below 2^24, so P is exact up to the
    # finalisation's FP32 rounding, whatever the rows' alignment
    import torch
    N, M, ld = 300, 130001, 130004
    U = (np.random.default_rng(shift).uniform(size=(N, M)) < 0.4).astype(np.float32)
    buf = torch.zeros(N * ld + 8, dtype=torch.float32, device="cuda")
    view = buf[shift:shift + N * ld].view(N, ld)[:, :M]
    view.copy_(_dev(U))
    o = H.full(view, mode="full", precision="bf16", want_P=True)
    H.sync()
    assert_close(to_np(o["P"]), O.inclusion_matrix(U), FP32_TOL, f"P, rows shifted by {shift}")


@pytest.mark.parametrize("sigma", [0.0, 0.2])
def test_fields(H, sigma):
    F = np.random.default_rng(7).normal(0.5, 0.3, (270, 120007)).astype(np.float32)
    o = H.from_fields(_dev(F), 0.5, sigma, mode="full", precision="split_bf16")
    H.sync()
    _check(o, O.iso_soft_mask(F, 0.5, sigma), None, f"fields sigma {sigma}")


def test_repeated_and_batched_calls_agree(H):
    # the flags of shared chunks are cleared for every launch, recorded ones included
    U = _dev(synth.random_soft(300, 400003, seed=9))
    one = H.full(U, mode="full", precision="split_bf16")
    items = [dict(data=U, mode="full", precision="split_bf16"), dict(data=U, mode="full", precision="bf16")]
    outs = None
    for _ in range(3):
        outs = H.batch(items, outs=outs)
    H.sync()
    np.testing.assert_array_equal(to_np(outs[0]["depth"]), to_np(one["depth"]))
