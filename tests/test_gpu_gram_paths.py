"""The two ways of the Gram of 257 to 512 members, clusters in one pass over the data and tiles over
staged operands: the same bits in every output, whichever is taken, for three and four row blocks,
full and partly filled, each precision, cell measures, every isovalue map, rows off the 16-byte
boundary, chunks that clusters share, batches and space-time steps; and a call whose operand planes
do not fit the handle's budget takes the clusters.

The masks have sigmoid tails, so that products summed in another order have other bits."""
import numpy as np
import pytest

from oracle import pid_oracle as O
from tests.helpers import FP32_TOL, GRAM_TOL, assert_close, to_np

pytestmark = pytest.mark.gpu

KEYS = ("depth", "in_in", "in_out", "rank", "P", "err_est")


@pytest.fixture(scope="module")
def handles():
    from paper_2512_15187_gb300 import binding, build
    build.build()
    hs = [binding.Handle(0) for _ in range(3)]
    for path, h in enumerate(hs):
        assert binding.load().pid_selftest_gram_path(h.h, path) == binding.PID_OK
    yield hs
    for h in hs:
        h.close()


def _masks(N, M, fields=False):
    import torch
    g = torch.Generator("cuda").manual_seed(N + M)
    s = torch.linspace(-1, 1, M, device="cuda").abs()
    c = 0.5 * torch.rand((N, 1), generator=g, device="cuda")
    width = 0.02 + 0.08 * torch.rand((N, 1), generator=g, device="cuda")
    x = (c - s) / width
    return 0.5 + 0.2 * x.clamp(-4, 4) if fields else torch.sigmoid(x)


def _shifted(U, shift):
    import torch
    N, M = U.shape
    ld = M + 3 if shift else (M + 3) // 4 * 4
    buf = torch.zeros(N * ld + 8, device="cuda")
    view = buf[shift:shift + N * ld].view(N, ld)[:, :M]
    view.copy_(U)
    return view


def _same(outs, what):
    for o in outs[1:]:
        for k in KEYS:
            if k in outs[0]:
                np.testing.assert_array_equal(to_np(outs[0][k]), to_np(o[k]), err_msg=f"{what} {k}")


@pytest.mark.parametrize("prec", ["bf16", "split_bf16", "fp8"])
@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("N,M,weighted", [(257, 120001, True), (300, 270000, False), (384, 262144, True),
                                          (391, 249985, False), (512, 230013, True), (512, 9000, False)])
def test_masks(handles, prec, shift, N, M, weighted):
    import torch
    U = _shifted(_masks(N, M), shift)
    w = torch.rand(M, device="cuda", generator=torch.Generator("cuda").manual_seed(1)) + 0.5 if weighted else None
    outs = [h.full(U, w, mode="full", precision=prec, want_P=prec != "fp8", want_err=True) for h in handles]
    for h in handles:
        h.sync()
    _same(outs, f"{prec} {N} x {M} shift {shift}")


@pytest.mark.parametrize("prec", ["bf16", "split_bf16", "fp8"])
@pytest.mark.parametrize("kind,superlevel,sigma", [("normal", False, 0.2), ("normal", True, 0.2), ("normal", False, 0.0),
                                                   ("normal", True, 0.0), ("uniform", False, 0.3),
                                                   ("uniform", True, 0.3), ("level", False, 0.4)])
@pytest.mark.parametrize("N,M,shift", [(270, 120007, 0), (390, 130000, 1)])
def test_fields(handles, prec, kind, superlevel, sigma, N, M, shift):
    F = _shifted(_masks(N, M, fields=True), shift)
    outs = [h.from_fields(F, 0.5, sigma, superlevel, mode="full", precision=prec, kind=kind) for h in handles]
    for h in handles:
        h.sync()
    _same(outs, f"{kind} {superlevel} {sigma} {prec}")
    ref = {"normal": lambda x: O.iso_soft_mask(x, 0.5, sigma, superlevel),
           "uniform": lambda x: O.iso_soft_mask_uniform(x, 0.5, sigma, superlevel),
           "level": lambda x: O.level_soft_mask(x, 0.5, sigma)}[kind]
    if shift == 0:
        want = O.pid(ref(to_np(F)), None)
        assert_close(to_np(outs[2]["in_in"]), want[0], FP32_TOL, "in_in")
        assert_close(to_np(outs[2]["depth"]), want[2], GRAM_TOL, "depth")


def test_batches(handles):
    data = [_masks(300, 150001), _masks(512, 131072), _masks(384, 200000), _masks(330, 120000)]
    items = [dict(data=U, mode="full", precision=p, want_P=p != "fp8") for U in data
             for p in ("bf16", "split_bf16", "fp8")]
    alone = [handles[0].full(i["data"], mode="full", precision=i["precision"], want_P=i["want_P"]) for i in items]
    handles[0].sync()
    for h in handles:
        outs = None
        for _ in range(3):                       # recorded, then replayed: the flags are cleared each time
            outs = h.batch(items, outs=outs)
        h.sync()
        for o, a, i in zip(outs, alone, items):
            _same([{k: a[k] for k in KEYS if k in a and k != "err_est"}, o], f"{i['data'].shape} {i['precision']}")


@pytest.mark.parametrize("prec", ["bf16", "split_bf16", "fp8"])
def test_spacetime(handles, prec):
    steps = [_masks(300, 120001) * f for f in (1.0, 0.75, 0.5)]
    outs = [h.spacetime(steps, mode="full", precision=prec) for h in handles]
    for h in handles:
        h.sync()
    _same(outs, f"space-time {prec}")


def test_budget_without_room_for_operand_planes():
    from paper_2512_15187_gb300 import binding
    U = _masks(300, 400000)                      # planes of 240 MB; tiles by the rule
    want = binding.Handle(0)
    o = want.full(U, mode="full", precision="bf16")
    want.sync()
    assert want.workspace_bytes() > 240 << 20
    tight = binding.Handle(0, hbm_budget_bytes=100 << 20)
    _same([o, tight.full(U, mode="full", precision="bf16")], "budget")
    _same([o, tight.batch([dict(data=U, mode="full", precision="bf16")])[0]], "budget, batch")
    tight.sync()
    assert tight.workspace_bytes() <= 100 << 20
