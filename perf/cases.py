"""The work that users have the solver do, as cases that can be timed and checked.

A case is one call of the library on one kind of grid: a device solve, a solve
from page-locked host buffers, a batch of uneven problems in one call, or the
Dirichlet potential alone.  Sizes are those of the named workloads (65^2, 129^3,
257^3, 513^3, the 33 ... 257 size classes of the batched workload, 258^3 as
given) and of the paper's refinement studies (panel counts that need padding).
`draw` gives more of the same ranges.
"""
import math

import numpy as np
import torch

import paper_2108_11871_gb300 as idp
from paper_2108_11871_gb300 import binding as _b

PRECISION = {"fp64": _b.IDP_PRECISION_FP64, "df32": _b.IDP_PRECISION_DF32,
             "bf16x3": _b.IDP_PRECISION_MIXED_BF16X3, "tf32x3": _b.IDP_PRECISION_MIXED_TF32X3}
BATCH_NODES = (33, 65, 97, 129, 193, 257)


def _case(call, sizes, density="gauss", order=6, precision="fp64", boundary_df32=False, exact_grid=False,
          tune=False, length0=1.0, name=None):
    c = dict(call=call, sizes=sizes, density=density, order=order, precision=precision,
             boundary_df32=boundary_df32, exact_grid=exact_grid, tune=tune, length0=length0)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the 2-D introductory solve: the smallest call, a chain of short launches
        _case("solve", "65x65", density="bump", name="bump_65x65"),
        # a fine 2-D solve with unequal sides
        _case("solve", "513x385", name="gauss_513x385"),
        # a small member of the batched family, solved by itself
        _case("solve", "33x65x97", name="gauss_33x65x97"),
        # the 3-D bump on a tuned plan, the paper's test density
        _case("solve", "129x129x129", density="bump", tune=True, name="bump_129"),
        # the refined 3-D solve at 4th order
        _case("solve", "193x193x193", order=4, name="gauss_193_order4"),
        # the precision sweep's grid in FP64
        _case("solve", "257x257x257", name="gauss_257"),
        # the large single solve, anisotropic mesh
        _case("solve", "513x513x513", length0=2.0, name="gauss_513"),
        # panel counts 100, 140, 74 as the convergence studies use them: padded grids
        _case("solve", "101x141x75", name="padded_101x141x75"),
        # double-float transforms
        _case("solve", "257x193x129", precision="df32", name="df32_257x193x129"),
        # tensor-core sine transforms, boundary in double-float: the fastest mode
        _case("solve", "257x257x257", precision="bf16x3", boundary_df32=True, name="bf16x3_257"),
        # a program whose data live in page-locked host memory
        _case("host", "129x129x129", density="bump", name="host_129"),
        # independent problems of uneven sizes in one call
        _case("batched", "33x65x129,129x97x193,65x65x65,193x129x33,97x97x97,257x129x65,33x193x65,129x129x129",
              name="batched_8"),
    ]


def draw(rng):
    def nodes(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def box(d, lo, hi):
        return "x".join(str(nodes(lo, hi)) for _ in range(d))

    kind = rng.choice(["solve2d", "solve3d", "solve3d", "solve3d", "reduced", "reduced", "exact", "phistar", "host",
                       "batched"])
    order = rng.choice([4, 6, 6, 6])
    density = rng.choice(["bump", "gauss"])
    length0 = rng.choice([1.0, 1.0, 2.0])
    if kind == "solve2d":
        return _case("solve", box(2, 17, 513), density, order)
    if kind == "reduced":
        p = rng.choice(["df32", "df32", "bf16x3", "tf32x3"])
        return _case("solve", box(3, 33, 257), density, order, p, p != "df32" and rng.random() < 0.5,
                     length0=length0)
    if kind == "exact":
        return _case("solve", box(3, 20, 140), density, order, rng.choice(["fp64", "bf16x3"]), exact_grid=True)
    if kind == "phistar":
        # a stage runs on the grid as given: sizes that need no padding
        return _case("phistar", "x".join(str(rng.choice(BATCH_NODES)) for _ in range(3)), density)
    if kind == "host":
        return _case("host", box(3, 17, 200), density, order)
    if kind == "batched":
        return _case("batched", ",".join("x".join(str(rng.choice(BATCH_NODES[:5])) for _ in range(3))
                                         for _ in range(rng.randint(2, 6))), "gauss", order)
    return _case("solve", box(3, 17, 380), density, order, length0=length0)


def _grids(case):
    return [tuple(int(v) for v in s.split("x")) for s in case["sizes"].split(",")]


def _box(case, d):
    if case["density"] == "bump":
        return [-1.0] * d, [1.0] * d
    return [0.0] * d, [float(case["length0"])] + [1.0] * (d - 1)


def _h(case, n):
    lo, hi = _box(case, len(n))
    return [(b - a) / (k - 1) for a, b, k in zip(lo, hi, n)]


def _step(t):
    """C-infinity step from 0 (t <= 0) to 1 (t >= 1)."""
    t = t.clamp(0.0, 1.0)
    a = torch.where(t > 0, torch.exp(-1.0 / t.clamp_min(1e-300)), torch.zeros_like(t))
    b = torch.where(t < 1, torch.exp(-1.0 / (1.0 - t).clamp_min(1e-300)), torch.zeros_like(t))
    return a / (a + b)


def _density(case, n, rng):
    """A smooth density that vanishes near the boundary, on every node."""
    d = len(n)
    lo, hi = _box(case, d)
    dev = torch.device("cuda")
    xs = []
    for s in range(d):
        shape = [1] * d
        shape[s] = n[s]
        x = lo[s] + torch.arange(n[s], dtype=torch.float64, device=dev) * ((hi[s] - lo[s]) / (n[s] - 1))
        xs.append(x.reshape(shape))
    if case["density"] == "bump":
        eps, p = (0.7, 10) if d == 3 else (0.8, 8)
        c = rng.uniform(-0.1, 0.1, size=d)
        u = sum((x - float(ci)) ** 2 for x, ci in zip(xs, c)) / eps ** 2
        return (1.0 - u).clamp_min(0.0).pow(p).contiguous()
    centres, sigma, amp = rng.uniform(0.3, 0.7, (6, d)), rng.uniform(0.04, 0.1, 6), rng.uniform(-1.0, 1.0, 6)
    out = torch.zeros(n, dtype=torch.float64, device=dev)
    for j in range(6):
        factor = float(amp[j])
        for s in range(d):
            c = lo[s] + centres[j, s] * (hi[s] - lo[s])
            factor = factor * torch.exp(-((xs[s] - float(c)) ** 2) / (2.0 * float(sigma[j]) ** 2))
        out += factor
    for s in range(d):
        xi = (xs[s] - lo[s]) / (hi[s] - lo[s])
        out *= torch.minimum(_step((xi - 0.15) / 0.15), _step((0.85 - xi) / 0.15))
    return out


def _densities(case, seed):
    return [_density(case, n, np.random.default_rng([seed, i])) for i, n in enumerate(_grids(case))]


def prepare(case, seed):
    plans = []
    for n in _grids(case):
        p = idp.create_plan(len(n), n, _h(case, n), case["order"], exact=case["exact_grid"])
        if case["precision"] != "fp64":
            idp.plan_set(p, _b.IDP_KEY_PRECISION, PRECISION[case["precision"]])
        if case["boundary_df32"]:
            idp.plan_set(p, _b.IDP_KEY_MIXED_BOUNDARY_DF32, 1)
        if case["tune"]:
            idp.plan_set(p, _b.IDP_KEY_AUTOTUNE, 1)
        plans.append(p)
    rho = _densities(case, seed)
    if case["call"] == "host":
        rho = [r.cpu().pin_memory() for r in rho]
        phi = [torch.empty_like(r).pin_memory() for r in rho]
    else:
        phi = [torch.empty_like(r) for r in rho]
    return dict(call=case["call"], plans=plans, rho=rho, phi=phi)


def run(state):
    call, plans, rho, phi = state["call"], state["plans"], state["rho"], state["phi"]
    if call == "batched":
        idp.solve_batched(plans, rho, phi)
        return phi
    if call == "host":
        idp.solve_host(plans[0], rho[0], phi[0])
    elif call == "phistar":
        idp.solve_stage(plans[0], _b.IDP_STAGE_PHISTAR, rho[0], phi[0])
    else:
        idp.solve(plans[0], rho[0], phi[0])
    return phi[0]


def work(case):
    """rho read and phi written once; the fast transforms of the method (2.5 log2(2M)
    operations a point for a sine pass, and the boundary's padded convolutions: for
    each face axis the real transforms of the lines, and a transform along the second
    axis and two real products for each slice)."""
    byte = flop = 0.0
    for n in _grids(case):
        d, pts = len(n), float(np.prod(n))
        lg = [math.log2(2 * (k - 1)) for k in n]
        byte += 16.0 * pts
        sine = {4: 3, 6: 4}[case["order"]] if case["call"] != "phistar" else 2
        flop += sine * pts * 2.5 * sum(lg)
        if d > 1 and case["call"] != "phistar":
            flop += 2 * pts * 2.5 * 2 * max(lg)
            if d == 3:
                flop += 3 * 2 * pts * (5.0 * max(lg) + 8.0)
    return {"bytes": byte, "flops": flop}


# ---- the same results from plain torch in 64 bits ---------------------------------


def _padded(M):
    """Panel counts 2^a in 16..512 and 3 2^a in 48..384 are solved as given, others on the next of these."""
    good = sorted([16 << a for a in range(6)] + [48 << a for a in range(4)])
    return next(m for m in good if m >= M)


def _along(a, m, axis):
    return torch.movedim(torch.tensordot(m, a, dims=([1], [axis])), 0, axis)


def _sines(a):
    """sum_i a_i sin(pi k i / M) along every axis of an interior array."""
    for s in range(a.dim()):
        M = a.shape[s] + 1
        k = np.arange(1, M, dtype=np.int64)
        m = torch.from_numpy(np.sin(np.pi * (np.outer(k, k) % (2 * M)) / M)).to(a.device)
        a = _along(a, m, s)
    return a


def _outer_sum(vs):
    d = len(vs)
    return sum(torch.from_numpy(v).cuda().reshape([-1 if t == s else 1 for t in range(d)]) for s, v in enumerate(vs))


def _inner(u, k=1):
    return u[tuple(slice(k, n - k) for n in u.shape)]


def _diff2(u, s, h):
    n = u.shape[s]
    return (u.narrow(s, 2, n - 2) - 2.0 * u.narrow(s, 1, n - 2) + u.narrow(s, 0, n - 2)) / (h * h)


def _cut(u, n, lost, to):
    for s in range(u.dim()):
        u = u.narrow(s, to - lost.count(s), n[s] - 2 * to)
    return u


def _boundary(rho, h):
    """G * rho on the boundary nodes by zero-padded convolutions, 0 inside."""
    n, d = rho.shape, rho.dim()
    out = torch.zeros_like(rho)
    if d == 1:
        i = torch.arange(1, n[0] - 1, device=rho.device, dtype=torch.float64)
        out[0] = 0.5 * h[0] ** 2 * (i * rho[1:-1]).sum()
        out[-1] = 0.5 * h[0] ** 2 * ((n[0] - 1 - i) * rho[1:-1]).sum()
        return out
    for a in range(d):
        rest = [s for s in range(d) if s != a]
        src = torch.movedim(rho, a, 0)
        long = [2 * (n[s] - 1) for s in rest]
        off = _outer_sum([(np.minimum(np.arange(2 * (n[s] - 1)), 2 * (n[s] - 1) - np.arange(2 * (n[s] - 1))) * h[s]) ** 2
                          for s in rest])
        np_, axes = n[a] - 2, tuple(range(1, d))
        lo = hi = 0.0
        chunk = max(1, (1 << 25) // int(np.prod(long)))
        keep = (slice(None),) + tuple(slice(1, n[s] - 1) for s in rest)

        def spectra(p0, p1):
            z = torch.zeros([p1 - p0] + [n[s] for s in rest], dtype=torch.float64, device=rho.device)
            z[keep] = src[p0:p1][keep]
            return torch.fft.rfftn(z, s=long, dim=axes)

        for p0 in range(1, np_ + 1, chunk):
            p1 = min(np_ + 1, p0 + chunk)
            r2 = (torch.arange(p0, p1, device=rho.device, dtype=torch.float64) * h[a]).square().reshape([-1] + [1] * (d - 1)) + off
            k = torch.fft.rfftn(-1.0 / (4.0 * math.pi * r2.sqrt()) if d == 3 else r2.log() / (4.0 * math.pi), dim=axes)
            lo = lo + (spectra(p0, p1) * k).sum(0)
            hi = hi + (spectra(n[a] - p1, n[a] - p0).flip(0) * k).sum(0)
        face = torch.movedim(out, a, 0)
        for i, acc in ((0, lo), (n[a] - 1, hi)):
            w = torch.fft.irfftn(acc, s=long, dim=tuple(range(d - 1)))
            face[i] = w[tuple(slice(0, n[s]) for s in rest)] * math.prod(h)
    return out


def _potential(rho, h, order, full=True):
    d, n = rho.dim(), rho.shape
    M = [k - 1 for k in n]
    scale = math.prod(2.0 / m for m in M)
    cont = _outer_sum([-((np.pi * np.arange(1, m) / (m * hs)) ** 2) for m, hs in zip(M, h)])
    star = _sines(scale * _sines(_inner(rho).contiguous()) / cont)
    if not full:
        out = torch.zeros_like(rho)
        _inner(out).copy_(star)
        return out
    u = _boundary(rho, h)
    if d == 1:
        t = torch.arange(n[0], device=rho.device, dtype=torch.float64) / M[0]
        u = u[0] * (1.0 - t) + u[-1] * t
        _inner(u).add_(star)
        return u
    lam = [-(4.0 / hs ** 2) * np.sin(np.pi * np.arange(1, m) / (2.0 * m)) ** 2 for m, hs in zip(M, h)]
    lam4 = _outer_sum(lam)
    rhs = sum(_cut(_diff2(u, s, h[s]), n, [s], 1) for s in range(d))
    for s in range(d):
        for r in range(s + 1, d):
            c = (h[s] ** 2 + h[r] ** 2) / 12.0
            zs = [np.zeros(m - 1) for m in M]
            ls, lr = list(zs), list(zs)
            ls[s], lr[r] = lam[s], lam[r]
            lam4 = lam4 + c * _outer_sum(ls) * _outer_sum(lr)
            rhs = rhs + c * _cut(_diff2(_diff2(u, r, h[r]), s, h[s]), n, [s, r], 1)
    _inner(u).copy_(_sines(scale * _sines(-rhs) / lam4))
    if order == 6:
        R = 0.0
        for s in range(d):
            for r in range(d):
                if r != s:
                    c = h[s] ** 4 / 240.0 + h[s] ** 2 * h[r] ** 2 / 144.0
                    R = R + c * _cut(_diff2(_diff2(_diff2(u, r, h[r]), s, h[s]), s, h[s]), n, [s, s, r], 2)
        for s in range(d):
            a = torch.movedim(R, s, 0)
            first = 4.0 * a[0] - 6.0 * a[1] + 4.0 * a[2] - a[3]
            last = 4.0 * a[-1] - 6.0 * a[-2] + 4.0 * a[-3] - a[-4]
            R = torch.movedim(torch.cat([first[None], a, last[None]]), 0, s)
        _inner(u).add_(_sines(scale * _sines(R) / lam4))
    _inner(u).add_(star)
    return u


def exact(case, seed):
    outs = []
    for n, rho in zip(_grids(case), _densities(case, seed)):
        h = _h(case, n)
        if case["exact_grid"]:
            big, off = n, [0] * len(n)
        else:
            big = [_padded(k - 1) + 1 for k in n]
            off = [(b - k) // 2 for b, k in zip(big, n)]
        wide = torch.zeros(tuple(big), dtype=torch.float64, device=rho.device)
        wide[tuple(slice(o + 1, o + k - 1) for o, k in zip(off, n))] = _inner(rho)
        phi = _potential(wide, h, case["order"], case["call"] != "phistar")
        phi = phi[tuple(slice(o, o + k) for o, k in zip(off, n))].contiguous()
        outs.append(phi.cpu() if case["call"] == "host" else phi)
    return outs if case["call"] == "batched" else outs[0]
