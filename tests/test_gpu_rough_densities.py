"""Boundary values of rough densities through the block fixed-point path (GPU): no further off than
FP64 transforms leave them.  Reference: the direct trapezoid sum at seeded boundary nodes.
"""
import numpy as np
import pytest

import workloads as w
from oracle import greens as ogreens

pytestmark = pytest.mark.gpu


def _error(n, rho, count):
    import torch
    import paper_2108_11871_gb300 as idp
    h = [1.0 / (max(n) - 1)] * len(n)
    idx = ogreens.boundary_indices(n)
    t = idx[np.random.default_rng(0).choice(len(idx), count, replace=False)]
    ref = ogreens.boundary_direct(rho, h, t)
    plan = idp.create_plan(len(n), n, h, 4, exact=max(n) == 300)
    r = torch.from_numpy(np.ascontiguousarray(rho)).cuda()
    out = torch.empty_like(r)
    idp.solve_stage(plan, idp.IDP_STAGE_BOUNDARY, r, out)
    torch.cuda.synchronize()
    return np.abs(out.cpu().numpy()[tuple(t.T)] - ref).max() / np.abs(ref).max()


@pytest.mark.parametrize("n", [(513, 513), (33, 513, 33), (33, 33, 513)], ids=lambda n: "x".join(map(str, n)))
def test_mean_errors_do_not_add_up_over_lines(n):
    # the spectra of the kernel, in FP64, are sums of up to 512 terms rounded at 2^-53 each:
    # 23 * 2^-53; errors of the transforms that add up over the lines and slices come on top
    assert _error(n, w.random_interior(n, seed=3), 200) <= 24 * 2.0 ** -53


def _density(kind, n):
    rho = np.zeros(n)
    noise = w.random_interior(n, seed=3)
    if kind == "noise":
        return noise
    mid = tuple(k // 2 for k in n)
    if kind == "line":
        rho[mid[0], mid[1]] = noise[mid[0], mid[1]]
    elif kind == "points":   # two large charges on faint noise
        rho = 1e-6 * noise
        rho[mid], rho[tuple(k // 3 for k in n)] = 1.0, -0.7
    elif kind == "plane":    # every frequency of one slice next to a face
        rho[1, 1:-1, 1:-1] = 1.0
    else:                    # one sign throughout: the sums reach their bounds
        rho[1:-1, 1:-1, 1:-1] = 1.0
    return rho


@pytest.mark.parametrize("n", [(193, 193, 193), (257, 257, 257), (385, 385, 33), (513, 513, 33), (300, 20, 25)],
                         ids=lambda n: "x".join(map(str, n)))
@pytest.mark.parametrize("kind", ["noise", "line", "points", "plane", "constant"])
def test_the_unit_follows_the_charge(n, kind):
    # The face passes' unit follows the sum of the line bounds of a pair of slices, within a factor of
    # two: where few lines are charged, and on noise, whose lines' spectra are far below their absolute sums, it is
    # no coarser than what FP64 would lose.  64 * 2^-53: the spectra's 23 (above), and as
    # much again for each of the two transforms.  Points: a point's spectrum does not fall, and the
    # FP64 spectra of the kernel alone leave 3e-14 of the largest value, 270 * 2^-53
    tol = (64 if kind != "points" else 400) * 2.0 ** -53
    assert _error(n, _density(kind, n), 60) <= tol


@pytest.mark.parametrize("n", [(33, 49, 17), (65, 65, 65), (49, 65)], ids=lambda n: "x".join(map(str, n)))
def test_sums_past_the_range_are_not_finite(n):
    # densities whose transforms overflow: a boundary value is the scaled one or not finite
    import torch
    import paper_2108_11871_gb300 as idp
    plan = idp.create_plan(len(n), n, [1.0 / (max(n) - 1)] * len(n), 4)

    def g(rho):
        r = torch.from_numpy(rho).cuda()
        out = torch.empty_like(r)
        idp.solve_stage(plan, idp.IDP_STAGE_BOUNDARY, r, out)
        torch.cuda.synchronize()
        return out.cpu().numpy()

    x = np.meshgrid(*[np.linspace(-1.0, 1.0, k) for k in n], indexing="ij")
    for rho in (np.maximum(0.0, 1.0 - sum(c * c for c in x)) ** 6, w.random_interior(n, seed=3)):
        base = g(rho)
        for power in range(1008, 1024):
            got = g(np.ldexp(rho, power))
            with np.errstate(over="ignore"):
                ref = np.ldexp(base, power)
            assert (~np.isfinite(got) | (got == ref)).all(), power
        assert not np.isfinite(got[ogreens.boundary_mask(n)]).any()


@pytest.mark.parametrize("n", [(129, 129, 129), (97, 65, 129), (193, 33, 65), (65, 65, 65)],
                         ids=lambda n: "x".join(map(str, n)))
@pytest.mark.parametrize("kind", ["noise", "sparse"])
def test_autotuning_leaves_the_bits(n, kind):
    # the sums over slices are the same integers for every number of chunks (odd or even), with
    # slices of zeros among them
    import torch
    import paper_2108_11871_gb300 as idp
    rho = w.random_interior(n, seed=3)
    if kind == "sparse":
        rho[5:9] = 0.0
        rho[20] = 0.0
        rho[:, 11:14] = 0.0
        rho[:, :, 7] = 0.0
    r = torch.from_numpy(rho).cuda()
    bits, chunks = set(), set()
    for tune in (0, 1):
        plan = idp.create_plan(3, n, [1.0 / (max(n) - 1)] * 3, 6)
        idp.plan_set(plan, idp.IDP_KEY_AUTOTUNE, tune)
        chunks.add(tuple(idp.plan_tuning(plan)["face_chunks"]))
        out = torch.empty_like(r)
        idp.solve(plan, r, out)
        torch.cuda.synchronize()
        bits.add(out.cpu().numpy().tobytes())
    print(n, chunks)
    assert len(bits) == 1
