"""The block fixed-point boundary path at the edges of its range (GPU): real FFTs,
face passes (3-D), inverse transforms, and the layer terms of the solution.

Tolerance: a density of random sign has a white spectrum, against which every pass is
off by a few 2^-53; the tables of the kernel spectra, FP64 on both sides, are off
by 2^-53 of their largest entry at every one of up to N = 512 frequencies of an axis, which
adds up to N 2^-53 = 6e-14 of g: 1e-12 leaves a factor of 16.  The correction u has its largest
value on the boundary and phi* stays below 1e-13 of its own, so phi gets 4e-12 (random errors
of 1e-12 of g on the boundary, put into the oracle's correction, moved phi by 0.9e-12 at most).
"""
import numpy as np
import pytest

import workloads as w
from oracle import greens as ogreens
from oracle import solve as osolve

pytestmark = pytest.mark.gpu

G_TOL, PHI_TOL = 1e-12, 4e-12
# (shape, exact): lengths 16 to 512, radix 3 and 6, unequal sides, one or two odd slices
# in the middle, rows that leave most of a block idle, and axes padded to the next length
GRIDS = [((17, 17), False), ((17, 513), False), ((513, 33), False), ((97, 49), False), ((385, 193), False),
         ((17, 17, 17), False), ((33, 17, 49), False), ((65, 97, 49), False), ((17, 129, 193), False),
         ((129, 17, 257), False), ((23, 41, 30), True), ((12, 70), True)]


def _h(n):
    return [1.0 / (max(n) - 1)] * len(n)


def _run(idp, n, rho, order=4, exact=False, stage=None):
    import torch
    plan = idp.create_plan(len(n), n, _h(n), order, exact=exact)
    r = torch.from_numpy(np.ascontiguousarray(rho)).cuda()
    out = torch.empty_like(r)
    if stage is None:
        idp.solve(plan, r, out)
    else:
        idp.solve_stage(plan, stage, r, out)
    torch.cuda.synchronize()
    return out.cpu().numpy()


def _mixed(n):
    # random signs, slices of very different size side by side, and an empty slice
    rho = w.random_interior(n, seed=12)
    rho[3] *= 1e-9
    rho[..., 5] *= 1e-5
    rho[:, 6] = 0.0
    return rho


@pytest.mark.parametrize("n,exact", GRIDS, ids=["x".join(map(str, n)) for n, _ in GRIDS])
def test_noise_matches_the_oracle(n, exact):
    import paper_2108_11871_gb300 as idp
    rho = _mixed(n)
    ref = ogreens.boundary_convolution(rho, _h(n))
    mask = ogreens.boundary_mask(n)
    got = _run(idp, n, rho, exact=exact, stage=idp.IDP_STAGE_BOUNDARY)
    assert np.abs(got - ref)[mask].max() <= G_TOL * np.abs(ref[mask]).max()
    phi = osolve.solve(rho, _h(n), 4, boundary="convolution")
    got = _run(idp, n, rho, exact=exact)
    assert np.abs(got - phi).max() <= PHI_TOL * np.abs(phi).max()


@pytest.mark.parametrize("n", [(49, 65), (33, 49, 17)], ids=["2d", "3d"])
@pytest.mark.parametrize("power", [-300, -31, 250])
def test_scaled_densities_give_the_scaled_bits(n, power):
    # every scale follows the density's exponent: nothing is cut off at a fixed size
    import paper_2108_11871_gb300 as idp
    rho = _mixed(n)
    base = _run(idp, n, rho, order=6)
    assert np.array_equal(_run(idp, n, np.ldexp(rho, power), order=6), np.ldexp(base, power))


@pytest.mark.parametrize("n", [(49, 65), (33, 49, 17)], ids=["2d", "3d"])
def test_no_charge_gives_zero_and_a_nan_every_node(n):
    import paper_2108_11871_gb300 as idp
    rho = np.zeros(n)
    assert not _run(idp, n, rho, order=6).any()
    rho = _mixed(n)
    rho[tuple(k // 3 for k in n)] = np.nan
    assert np.isnan(_run(idp, n, rho, order=6)).all()


def test_rounding_has_no_bias():
    # a product that rounds one way is a bias, which the lowest frequency adds up over lines and
    # slices (factors 2^-62 below 1 gave 4e-14 here).  Unbiased: the face pass's unit is 2^-61
    # of the bound 2 * 128 * 128 on a column's absolute sum, 1e-15 of a coefficient of random
    # signs (about 13), a few units in all: 1e-14 for the largest error
    import paper_2108_11871_gb300 as idp
    n = (129, 129, 129)
    rho = w.random_interior(n, seed=3)
    idx = ogreens.boundary_indices(n)
    t = idx[np.random.default_rng(0).choice(len(idx), 40, replace=False)]
    ref = ogreens.boundary_direct(rho, _h(n), t)
    got = _run(idp, n, rho, stage=idp.IDP_STAGE_BOUNDARY)[tuple(t.T)]
    assert np.abs(got - ref).max() <= 1e-14 * np.abs(ref).max()
