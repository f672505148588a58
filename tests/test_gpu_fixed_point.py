"""The block fixed-point sine passes at the edges of their range (GPU).

A pass holds a line in 64-bit integers on a power-of-two scale taken from the
line's absolute sum, so that a density times a power of two has to give the same
bits times that power, whatever the exponent, and a line of any size has to agree
with the oracle.  Tolerance: a value is off by a few units of 2^-58 of its line's
absolute sum per pass, at most 2^-49 of the largest output for a line of 511 equally
large values of random sign; three forward and three inverse passes stay below 1e-13.
"""
import numpy as np
import pytest

import workloads as w
from oracle import dst as odst

pytestmark = pytest.mark.gpu

TOL = 1e-13
GRIDS = [(17, 33), (65, 49), (129, 97), (193, 257), (385, 513), (17, 25, 49), (33, 129, 17)]


def _phistar(idp, n, h, rho):
    import torch
    plan = idp.create_plan(len(n), n, h, 6, exact=True)
    r = torch.from_numpy(np.ascontiguousarray(rho)).cuda()
    out = torch.empty_like(r)
    idp.solve_stage(plan, idp.IDP_STAGE_PHISTAR, r, out)
    torch.cuda.synchronize()
    return out.cpu().numpy()


def _h(n):
    return [1.0 / (k - 1) for k in n]


@pytest.mark.parametrize("n", GRIDS, ids=lambda n: "x".join(map(str, n)))
def test_noise_lines_match_the_oracle(n):
    import paper_2108_11871_gb300 as idp
    rho = w.random_interior(n, seed=5)
    ref = odst.phi_star(rho, _h(n))
    got = _phistar(idp, n, _h(n), rho)
    assert np.abs(got - ref).max() <= TOL * np.abs(ref).max()


@pytest.mark.parametrize("power", [-800, -40, 300, 900])
def test_scaled_densities_give_the_scaled_bits(power):
    import paper_2108_11871_gb300 as idp
    n = (33, 49, 65)
    rho = w.random_interior(n, seed=6)
    rho[5] *= 1e-20          # lines of very different size side by side
    rho[:, 7] = 0.0
    base = _phistar(idp, n, _h(n), rho)
    got = _phistar(idp, n, _h(n), np.ldexp(rho, power))
    assert np.array_equal(got, np.ldexp(base, power))


def test_densities_next_to_the_smallest_numbers():
    # lines whose unit is below the smallest normal number
    import paper_2108_11871_gb300 as idp
    n = (33, 65)
    rho = w.random_interior(n, seed=8)
    ref = odst.phi_star(rho, _h(n))
    got = np.ldexp(_phistar(idp, n, _h(n), np.ldexp(rho, -985)), 985)
    assert np.abs(got - ref).max() <= TOL * np.abs(ref).max()


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_a_value_that_is_not_finite_reaches_every_node(bad):
    import paper_2108_11871_gb300 as idp
    n = (33, 33, 65)
    rho = w.random_interior(n, seed=7)
    rho[9, 20, 31] = bad
    got = _phistar(idp, n, _h(n), rho)
    assert np.isnan(got[1:-1, 1:-1, 1:-1]).all()
    assert not got[0].any()
