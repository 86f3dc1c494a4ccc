"""A call's results are the same bits alone, in a batch of its like, in a batch with larger
ensembles and among other requests of a server, at the member and chunk counts where the
finalisation splits an ensemble over one CTA or several.

The masks have sigmoid tails, so that a member's chunk sums span many orders of magnitude and a
sum in another order has other last bits."""
import numpy as np
import pytest

from tests.helpers import to_np

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def H():
    from paper_2512_15187_gb300 import binding, build
    build.build()
    h = binding.Handle(0)
    yield h
    h.close()


def _masks(N, M):
    rng = np.random.default_rng(N + M)
    s = np.abs(np.linspace(-1, 1, M))
    c, width = 0.5 * rng.random((N, 1)), 0.01 + 0.02 * rng.random((N, 1))
    return (1.0 / (1.0 + np.exp(np.clip((s - c) / width, -80, 80)))).astype(np.float32)


def _dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _same(a, b, what):
    for k in ("depth", "in_in", "in_out", "rank", "P"):
        if k in a and k in b:
            np.testing.assert_array_equal(to_np(a[k]), to_np(b[k]), err_msg=f"{what} {k}")


SHAPES = [(5, 3000), (8, 300000), (16, 65536), (20, 16384), (32, 8192), (33, 16384), (40, 5000), (100, 20000)]


@pytest.mark.parametrize("prec", ["bf16", "split_bf16", "fp8"])
def test_gram_items(H, prec):
    data = [_dev(_masks(*s)) for s in SHAPES]
    kw = dict(mode="full", precision=prec, want_P=prec != "fp8")
    alone = [H.full(U, **kw) for U in data]
    H.sync()
    for name, pick in (("small", [0, 2, 3, 4]), ("one", [3]), ("mixed", list(range(len(SHAPES)))),
                       ("repeated", [2, 3] * 40)):
        outs = H.batch([dict(data=data[k], **kw) for k in pick])
        H.sync()
        for o, k in zip(outs, pick):
            _same(o, alone[k], f"{SHAPES[k]} in the {name} batch")


@pytest.mark.parametrize("mode", ["mean", "linear"])
def test_streamed_items(H, mode):
    shapes = SHAPES + [(1, 700), (256, 30000), (300, 5000), (512, 9000)]
    data = [_dev(_masks(*s)) for s in shapes]
    alone = [H.mean(U) if mode == "mean" else H.full(U, mode="linear") for U in data]
    H.sync()
    for pick in (list(range(len(shapes))), [0, 1, 2] * 20, [0, 2, 3] * 120, ([0, 2, 3] * 3 + [9]) * 40,
                 list(range(len(shapes))) * 30):
        outs = H.batch([dict(data=data[k], mode=mode) for k in pick])
        H.sync()
        for o, k in zip(outs, pick):
            _same(o, alone[k], f"{shapes[k]} in a batch of {len(pick)}")


def test_served_mix(H):
    from paper_2512_15187_gb300 import binding as B
    data = [_masks(*s) for s in SHAPES]
    alone = [H.full(_dev(U), mode="full", precision="split_bf16") for U in data]
    H.sync()
    srv = B.Server(max_inflight=2, max_batch=16)
    try:
        ids = [srv.register(U) for U in data]
        for pick in ([3], list(range(len(SHAPES))) * 3):
            tickets = [(k, srv.submit(ids[k], "full", "split_bf16")) for k in pick]
            for k, t in tickets:
                o = srv.wait(t, SHAPES[k][0])
                for f in ("depth", "in_in", "in_out", "rank"):
                    np.testing.assert_array_equal(o[f], to_np(alone[k][f]), err_msg=f"{SHAPES[k]} {f}")
    finally:
        srv.stop()


# eight, four, two and one CTA per ensemble (152 SMs); 256 members' rows need two
@pytest.mark.parametrize("count", [10, 30, 60, 120, 320])
@pytest.mark.parametrize("N,M", [(33, 6000), (100, 4096), (225, 2048), (256, 2048)])
def test_many_gram_items(H, count, N, M):
    U = _dev(_masks(N, M))
    alone = H.full(U, mode="full", precision="split_bf16", want_P=True)
    outs = H.batch([dict(data=U, mode="full", precision="split_bf16", want_P=True)] * count)
    H.sync()
    for o in outs:
        _same(o, alone, f"{N} x {M}, {count} items")


# a Gram item takes a PID-mean or exact item's sums over the same masks: IN_in is bitwise the sibling's
@pytest.mark.parametrize("prec", ["bf16", "split_bf16", "fp8"])
@pytest.mark.parametrize("mode", ["mean", "linear"])
def test_in_in_of_a_sibling(H, prec, mode):
    for shape in SHAPES:
        U = _dev(_masks(*shape))
        a, b = H.batch([dict(data=U, mode=mode), dict(data=U, mode="full", precision=prec)])
        H.sync()
        np.testing.assert_array_equal(to_np(a["in_in"]), to_np(b["in_in"]), err_msg=f"{shape} {prec}")
        np.testing.assert_array_equal(to_np(a["mass"]), to_np(b["mass"]), err_msg=f"{shape} {prec}")
