"""The workloads that the library's speed is measured on.

Each case is one call that a user's program makes through the public binding
(paper_2512_15187_gb300.binding), at the sizes of the benchmark's workloads and of the
tests, from the smallest call to multi-gigabyte ensembles. `draw` gives further cases of the
same ranges. Inputs follow the recipes of the paper's workloads and are made here with plain
torch on the device, from the seed alone.

A state holds what a program has in hand before the call: the input tensors on the device
and a library handle (with the output tensors of a batch once it ran, which a program that
repeats the batch passes again).

Outputs: depths, inclusion fractions and ranks as the call returns them, with the inclusion
matrix where it is asked for. The Gram's raw error estimate is left out: it is the
difference of two nearly equal sums, a diagnostic of the rounding rather than a result.
"""
import math

import torch

from paper_2512_15187_gb300 import binding

ISO_MU, ISO_SIGMA = 0.5, 0.05      # isovalue ~ Normal(0.5, 0.05), the 2D fields workload


# ---- cases -----------------------------------------------------------------------------

def listed():
    return [
        # One small 2D ensemble of soft ellipses, PID-mean: the smallest call, as an
        # interactive tool makes it; launches and latency count.
        {"name": "ellipses_mean_20x128sq", "path": "mean", "data": "ellipses",
         "members": 20, "side": 128},
        # The same ensemble through the tensor-core Gram, with the inclusion matrix (for
        # clustering or per-group depths).
        {"name": "ellipses_gram_20x128sq", "path": "gram", "data": "ellipses",
         "members": 20, "side": 128, "precision": "bf16", "matrix": True},
        # One ensemble of 2D scalar fields with an uncertain isovalue: the map fused in front
        # of PID-mean.
        {"name": "fields_mean_64x512sq", "path": "fields_mean", "data": "fields",
         "members": 64, "side": 512},
        # Eight such ensembles (time steps, levels) in one replayed batch, exact full PID.
        {"name": "fields_batch_8x64x512sq", "path": "fields_batch", "data": "fields",
         "members": 64, "side": 512, "ensembles": 8},
        # A non-Cartesian grid: scattered points with cell measures, exact full PID.
        {"name": "disk_linear_128x1M", "path": "linear", "data": "disk",
         "members": 128, "cells": 1 << 20},
        # A large 3D ensemble (smoke plumes), PID-mean: one pass over 5.7 GB.
        {"name": "plume_mean_200x192cubed", "path": "mean", "data": "plume",
         "members": 200, "side": 192},
        # One time step of the 3D plume batch: PID-mean, and full PID with E4M3 and with
        # split-BF16 operands, over the same masks in one replayed batch.
        {"name": "plume_step_200x128cubed", "path": "step", "data": "plume",
         "members": 200, "side": 128},
        # A large ensemble's inclusion matrix at the tight precision (row-block-tiled Gram).
        {"name": "gram_split_512x1M", "path": "gram", "data": "disk",
         "members": 512, "cells": 1 << 20, "precision": "split_bf16", "matrix": True},
        # Uneven ensembles in one replayed batch, PID-mean and exact full PID of each, rows
        # as long as their cell counts (most of them not 16-byte aligned).
        {"name": "uneven_batch", "path": "uneven", "data": "uniform",
         "shapes": "300x1000003 63x1571042 441x90001 128x400004 17x25001"},
        # The scalability study: many members on a coarse 3D grid, PID-mean.
        {"name": "many_members_mean_10000x50cubed", "path": "mean", "data": "ellipsoids",
         "members": 10000, "side": 50},
        # Contour boxplot bands of one large ensemble of fields, from its ranks.
        {"name": "bands_64x2048sq", "path": "bands", "data": "fields",
         "members": 64, "side": 2048},
        # The isovalue map alone: soft masks of an ensemble of fields, stored.
        {"name": "soft_masks_64x2048sq", "path": "soft_masks", "data": "fields",
         "members": 64, "side": 2048},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    path = rng.choice(["mean", "linear", "gram", "gram", "fields_mean", "fields_batch", "step",
                       "uneven", "many", "bands", "soft_masks"])
    if path == "mean":
        if rng.random() < 0.5:
            return {"path": "mean", "data": "ellipses", "members": _log_int(rng, 8, 500),
                    "side": _log_int(rng, 64, 1024)}
        return {"path": "mean", "data": "plume", "members": rng.randint(16, 256),
                "side": _log_int(rng, 32, 160)}
    if path == "linear":
        if rng.random() < 0.5:
            return {"path": "linear", "data": "disk", "members": rng.randint(16, 256),
                    "cells": _log_int(rng, 1 << 14, 1 << 20)}
        return {"path": "linear", "data": "ellipses", "members": _log_int(rng, 8, 500),
                "side": _log_int(rng, 64, 1024)}
    if path == "gram":
        return {"path": "gram", "data": "disk", "members": _log_int(rng, 16, 512),
                "cells": _log_int(rng, 1 << 13, 1 << 20),
                "precision": rng.choice(["bf16", "split_bf16", "fp8"]),
                "matrix": rng.random() < 0.5}
    if path == "fields_mean":
        return {"path": "fields_mean", "data": "fields", "members": _log_int(rng, 8, 256),
                "side": _log_int(rng, 96, 1024)}
    if path == "fields_batch":
        return {"path": "fields_batch", "data": "fields", "members": rng.randint(16, 96),
                "side": _log_int(rng, 96, 512), "ensembles": rng.randint(2, 10)}
    if path == "step":
        return {"path": "step", "data": "plume", "members": rng.randint(16, 256),
                "side": _log_int(rng, 32, 128)}
    if path == "uneven":
        n = rng.randint(2, 5)
        shapes = [(rng.randint(10, 500), _log_int(rng, 64 ** 2, 1 << 20)) for _ in range(n)]
        while sum(N * M for N, M in shapes) > 6e8:      # no more than the largest listed batch
            shapes.remove(max(shapes, key=lambda s: s[0] * s[1]))
        return {"path": "uneven", "data": "uniform",
                "shapes": " ".join("%dx%d" % s for s in shapes)}
    if path == "many":
        members = _log_int(rng, 600, 20000)
        most = int((1.25e9 / members) ** (1 / 3))       # no more than 5 GB
        return {"path": "mean", "data": "ellipsoids", "members": members,
                "side": rng.randint(24, min(50, most))}
    if path == "bands":
        return {"path": "bands", "data": "fields", "members": _log_int(rng, 8, 256),
                "side": _log_int(rng, 128, 1024)}
    return {"path": "soft_masks", "data": "fields", "members": _log_int(rng, 8, 256),
            "side": _log_int(rng, 128, 1024), "bf16": rng.random() < 0.5}


# ---- inputs ----------------------------------------------------------------------------

def _generator(seed, salt=0):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 1009 + salt)


def _rand(shape, g):
    return torch.rand(shape, generator=g, device="cuda")


def _ellipses(N, side, g):
    """Soft ellipses on side^2 cells: centre within 8% of the middle, semi-axes 20 to 35% of
    the side, any rotation, edge width 1 to 3% of the side; u = sigmoid((1 - s) r / width)."""
    p = _rand((N, 6, 1), g)
    t = (torch.arange(side, device="cuda", dtype=torch.float32) + 0.5) / side
    yy, xx = (v.reshape(1, -1) for v in torch.meshgrid(t, t, indexing="ij"))
    out = torch.empty((N, side * side), device="cuda")
    for i in range(0, N, 32):
        q = p[i:i + 32]
        dy, dx = yy - (0.42 + 0.16 * q[:, 0]), xx - (0.42 + 0.16 * q[:, 1])
        a, b, th = 0.2 + 0.15 * q[:, 2], 0.2 + 0.15 * q[:, 3], math.pi * q[:, 4]
        u = (torch.cos(th) * dx + torch.sin(th) * dy) / a
        v = (torch.cos(th) * dy - torch.sin(th) * dx) / b
        s = torch.sqrt(u * u + v * v)
        out[i:i + 32] = torch.sigmoid((1.0 - s) * torch.sqrt(a * b) / (0.01 + 0.02 * q[:, 5]))
    return out


def _fields(N, side, g):
    """Scalar fields: 32 separable Gaussian bumps of amplitude N(1, 0.3) and width 4 to 12%
    of the side, plus noise of standard deviation 0.05, less a level that leaves the
    isovalue inside the field's range."""
    t = torch.arange(side, device="cuda", dtype=torch.float32) / side
    out = torch.empty((N, side * side), device="cuda")
    for i in range(0, N, 64):
        n = min(64, N - i)
        c, amp, sd = _rand((n, 2, 32, 1), g), torch.randn((n, 32, 1), generator=g, device="cuda"), \
            0.04 + 0.08 * _rand((n, 32, 1), g)
        gy = torch.exp(-((t - c[:, 0]) ** 2) / (2 * sd ** 2)) * (1.0 + 0.3 * amp)
        gx = torch.exp(-((t - c[:, 1]) ** 2) / (2 * sd ** 2))
        F = torch.bmm(gy.transpose(1, 2), gx).reshape(n, -1)
        F += 0.05 * torch.randn(F.shape, generator=g, device="cuda")
        out[i:i + n] = F - 0.25
    return out


def _disk(N, M, g):
    """Perturbed radial masks on M scattered points of the unit disk, 8 Fourier modes; cell
    measures log-uniform over two decades, summing to pi."""
    r, th = torch.sqrt(_rand((M,), g)), 2 * math.pi * _rand((M,), g)
    w = 10.0 ** (2 * _rand((M,), g))
    w = w * (math.pi / w.sum())
    k = torch.arange(1, 9, device="cuda", dtype=torch.float32)
    coef = torch.randn((N, 2, 8), generator=g, device="cuda") / k
    out = torch.empty((N, M), device="cuda")
    for i in range(0, N, 32):
        q = coef[i:i + 32]
        xi = sum(q[:, 0, j:j + 1] * torch.cos((j + 1) * th) + q[:, 1, j:j + 1] * torch.sin((j + 1) * th)
                 for j in range(8))
        xi = xi / xi.abs().amax(dim=1, keepdim=True)
        out[i:i + 32] = 0.5 * (1.0 + torch.tanh((0.5 + 0.1 * xi - r) / 0.02))
    return out, w


def _plume(N, R, g):
    """Smoke-plume-like masks on R^3 cells: a cone displaced by three octaves of trilinear
    value noise, u = sigmoid((radius(z) - rho + 0.08 noise) / 0.02)."""
    t = torch.linspace(0, 1, R, device="cuda")
    z = t.view(R, 1, 1)
    rho = torch.sqrt((t.view(1, R, 1) - 0.5) ** 2 + (t.view(1, 1, R) - 0.5) ** 2)
    base = (0.04 + 0.25 * z) * torch.clamp((0.8 - z) / 0.08, 0.0, 1.0) - rho
    out = torch.empty((N, R ** 3), device="cuda")
    step = max(1, (1 << 25) // R ** 3)
    for i in range(0, N, step):
        n = min(step, N - i)
        noise = 0.0
        for o in range(3):
            lat = 2.0 * _rand((n, 1, 4 * 2 ** o + 1, 4 * 2 ** o + 1, 4 * 2 ** o + 1), g) - 1.0
            noise = noise + 0.5 ** o * torch.nn.functional.interpolate(
                lat, size=(R, R, R), mode="trilinear", align_corners=True)[:, 0]
        out[i:i + n] = torch.sigmoid((base + 0.08 * noise) / 0.02).reshape(n, -1)
    return out


def _ellipsoids(N, R, g):
    """Soft ellipsoids in the unit cube on R^3 cells, a fifth of them outliers."""
    c = 0.5 + 0.02 * torch.randn((N, 3), generator=g, device="cuda")
    a = 0.25 + 0.015 * torch.randn((N, 3), generator=g, device="cuda")
    far = N // 5
    if far:
        c[-far:] = 0.5 + 0.08 * torch.randn((far, 3), generator=g, device="cuda")
        a[-far:] = 0.12 + 0.26 * _rand((far, 3), g)
    t = (torch.arange(R, device="cuda", dtype=torch.float32) + 0.5) / R
    out = torch.empty((N, R ** 3), device="cuda")
    step = max(1, (1 << 26) // R ** 3)
    for i in range(0, N, step):
        sl = slice(i, min(N, i + step))
        z, y, x = (((t - c[sl, k:k + 1]) / a[sl, k:k + 1]) ** 2 for k in range(3))
        s2 = z[:, :, None, None] + y[:, None, :, None] + x[:, None, None, :]
        out[sl] = torch.sigmoid((1.0 - torch.sqrt(s2)) / 0.05).reshape(s2.shape[0], -1)
    return out


def _shapes(case):
    if "shapes" in case:
        return [tuple(int(v) for v in s.split("x")) for s in case["shapes"].split()]
    M = case["cells"] if "cells" in case else case["side"] ** (3 if case["data"] in ("plume", "ellipsoids") else 2)
    return [(case["members"], M)] * case.get("ensembles", 1)


def _inputs(case, seed):
    """[(data [N, M], cell measures [M] or None)] of the case's ensembles."""
    got = []
    for e, (N, M) in enumerate(_shapes(case)):
        g = _generator(seed, e)
        if case["data"] == "disk":
            got.append(_disk(N, M, g))
        elif case["data"] == "uniform":
            got.append((_rand((N, M), g), None))
        else:
            make = {"ellipses": _ellipses, "fields": _fields, "plume": _plume, "ellipsoids": _ellipsoids}
            got.append((make[case["data"]](N, case["side"], g), None))
    return got


# ---- one pass --------------------------------------------------------------------------

def prepare(case, seed):
    data = _inputs(case, seed)
    state = {"case": case, "data": data, "handle": binding.Handle(0)}
    iso = (ISO_MU, ISO_SIGMA, 0)
    if case["path"] == "fields_batch":
        state["items"] = [dict(data=F, iso=iso, mode="linear") for F, _ in data]
    elif case["path"] == "step":
        U = data[0][0]
        state["items"] = [dict(data=U, mode="mean"), dict(data=U, mode="full", precision="fp8"),
                          dict(data=U, mode="full", precision="split_bf16")]
    elif case["path"] == "uneven":
        state["items"] = [dict(data=U, mode=mode) for U, _ in data for mode in ("mean", "linear")]
    elif case["path"] == "bands":
        # the ranks of an earlier depth call
        state["rank"] = torch.randperm(data[0][0].shape[0], generator=_generator(seed, 99),
                                       device="cuda").int()
    return state


def run(state):
    case, h = state["case"], state["handle"]
    path = case["path"]
    if "items" in state:
        state["outs"] = h.batch(state["items"], outs=state.get("outs"))
        return [{k: v for k, v in o.items() if k != "err_est"} for o in state["outs"]]
    x, w = state["data"][0]
    if path == "mean":
        return h.mean(x, w)
    if path == "linear":
        return h.full(x, w, mode="linear")
    if path == "gram":
        o = h.full(x, w, mode="full", precision=case["precision"], want_P=case["matrix"])
        return {k: v for k, v in o.items() if k != "err_est"}
    if path == "fields_mean":
        return h.from_fields(x, ISO_MU, ISO_SIGMA, mode="mean")
    if path == "bands":
        return h.contour_bands(x, state["rank"], 0.5, 0.5, iso=(ISO_MU, ISO_SIGMA, 0))
    return h.soft_masks(x, ISO_MU, ISO_SIGMA, dtype=torch.bfloat16 if case.get("bf16") else None)


# ---- the work a pass cannot do without -------------------------------------------------

def work(case):
    path = case["path"]
    size = flops = 0
    for N, M in _shapes(case):
        pairs = N * (N + 1) * M               # multiply-adds of the symmetric Gram
        size += 4 * N * M + (4 * M if case["data"] == "disk" else 0) + 28 * N
        if path == "mean":
            flops += 4 * N * M                # column sum, mass, product with the mean contour
        elif path == "linear":
            flops += 7 * N * M                # and the product with the second contour
        elif path == "fields_mean":
            flops += 24 * N * M               # the isovalue map takes about 20 per element
        elif path == "fields_batch":
            flops += 27 * N * M
        elif path == "uneven":
            size += 44 * N + 16 * N
            flops += 7 * N * M
        elif path == "gram":
            size += 8 * N * N if case["matrix"] else 0
            flops += pairs * (3 if case["precision"] == "split_bf16" else 1)
        elif path == "step":
            size += 2 * 28 * N + 3 * 16 * N
            flops += 4 * pairs + 4 * N * M
        elif path == "bands":
            size += M - 24 * N
            flops += N * M
        else:
            size += (2 if case.get("bf16") else 4) * N * M - 28 * N
            flops += 20 * N * M
    return {"bytes": size, "flops": flops}


# ---- the same results in 64 bits -------------------------------------------------------

def _mask64(F):
    return 0.5 * torch.special.erfc((F.double() - ISO_MU) / (ISO_SIGMA * math.sqrt(2.0)))


def _sums64(x, w, is_field, want_gram):
    """Masses, A_i = sum_x w u_i ubar and, on request, the Gram sum_x w u_i u_j."""
    N, M = x.shape
    m = torch.zeros(N, dtype=torch.float64, device="cuda")
    A = torch.zeros_like(m)
    G = torch.zeros((N, N), dtype=torch.float64, device="cuda") if want_gram else None
    step = max(1, (1 << 28) // N)
    for c in range(0, M, step):
        u = _mask64(x[:, c:c + step]) if is_field else x[:, c:c + step].double()
        wu = u if w is None else u * w[c:c + step].double()
        m += wu.sum(dim=1)
        A += wu @ u.mean(dim=0)
        if want_gram:
            G += wu @ u.T
    return m, A, G


def _ratio(a, b):
    return torch.where(b > 0, a / torch.where(b > 0, b, torch.ones_like(b)), torch.zeros_like(a))


def _out_linear64(x, w, is_field, m):
    """(1/N) sum_j (u_j subset_p u_i) = sum_x w u_i (1/N) sum_j u_j / m_j."""
    N, M = x.shape
    c = _ratio(torch.ones_like(m), m) / N
    out = torch.zeros_like(m)
    step = max(1, (1 << 28) // N)
    for k in range(0, M, step):
        u = _mask64(x[:, k:k + step]) if is_field else x[:, k:k + step].double()
        wu = u if w is None else u * w[k:k + step].double()
        out += wu @ (c @ u)
    return out


def _depths64(x, w, is_field, full, matrix=False, extras=False):
    m, A, G = _sums64(x, w, is_field, matrix)
    in_in, mean_out = _ratio(A, m), _ratio(A, m.mean().expand_as(A))
    in_out = _out_linear64(x, w, is_field, m) if full else mean_out
    o = {"depth": torch.minimum(in_in, in_out), "in_in": in_in, "in_out": in_out, "rank": None}
    if matrix:
        o["P"] = _ratio(G, m[:, None].expand_as(G))
    if extras:
        o["mass"], o["mean_depth"] = m, torch.minimum(in_in, mean_out)
    return o


def exact(case, seed):
    path = case["path"]
    if path == "bands":
        return None      # whole numbers
    data = _inputs(case, seed)
    x, w = data[0]
    if path == "soft_masks":
        return _mask64(x)
    if path == "mean":
        return _depths64(x, w, False, False)
    if path == "linear":
        return _depths64(x, w, False, True)
    if path == "gram":
        return _depths64(x, w, False, True, matrix=case["matrix"])
    if path == "fields_mean":
        return _depths64(x, w, True, False)
    if path == "fields_batch":
        return [_depths64(F, None, True, True, extras=True) for F, _ in data]
    if path == "step":
        return [_depths64(x, None, False, full, extras=True) for full in (False, True, True)]
    return [_depths64(U, None, False, full, extras=True) for U, _ in data for full in (False, True)]
