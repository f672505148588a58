"""The boundary values and the correction u1 that a plan's solve uses, in every precision mode (GPU),
against the oracle: FP64 and double-float FFTs in the tensor-core modes, fixed point in the others.
"""
import numpy as np
import pytest

import workloads as w
from oracle import greens as ogreens
from oracle import harmonic as oharm

pytestmark = pytest.mark.gpu

# face transforms of length 2 * 16 to 2 * 512, radix 3 among them, along each of the axes
GRIDS = [(513, 513), (385, 193), (97, 49), (65, 97, 49), (17, 129, 193), (129, 17, 257), (385, 17, 33), (17, 385, 33),
         (513, 33, 17), (33, 513, 17)]
# the kernel spectra in FP64 add up 512 roundings of 2^-53 per axis (6e-14 of g), with a factor of
# 16; double-float numbers carry 48 bits, 32 times the rounding, of which the factor is left out
G_TOL, DD_TOL = 1e-12, 4e-12


def _case(n):
    h = [1.0 / (max(n) - 1)] * len(n)
    x = np.meshgrid(*[np.linspace(-1.0, 1.0, k) for k in n], indexing="ij")
    rho = np.maximum(0.0, 1.0 - sum(c * c for c in x)) ** 4 * (1.0 + np.sin(5.0 * x[0] + 3.0 * x[1]))
    rho += 0.05 * w.random_interior(n, seed=4)
    return h, rho


def _run(idp, plan, rho, stage=None):
    import torch
    r = torch.from_numpy(np.ascontiguousarray(rho)).cuda()
    out = torch.empty_like(r)
    if stage is None:
        idp.solve(plan, r, out)
    else:
        idp.solve_stage(plan, stage, r, out)
    torch.cuda.synchronize()
    idp.plan_status(plan)
    return out.cpu().numpy()


@pytest.mark.parametrize("n", GRIDS, ids=lambda n: "x".join(map(str, n)))
def test_boundary_and_correction_of_a_solve(n):
    import paper_2108_11871_gb300 as idp
    h, rho = _case(n)
    parts = {}
    ref = ogreens.boundary_convolution(rho, h)
    oharm.harmonic_correction(ref, h, 4, parts)
    mask, top = ogreens.boundary_mask(n), np.abs(ref).max()
    got = {}
    for mode, bdd in (("FP64", 0), ("DF32", 0), ("MIXED_BF16X3", 0), ("MIXED_TF32X3", 0), ("MIXED_BF16X3", 1)):
        plan = idp.create_plan(len(n), n, h, 6)
        idp.plan_set(plan, idp.IDP_KEY_PRECISION, getattr(idp, "IDP_PRECISION_" + mode))
        idp.plan_set(plan, idp.IDP_KEY_MIXED_BOUNDARY_DF32, bdd)
        phi, u1 = _run(idp, plan, rho), _run(idp, plan, rho, idp.IDP_STAGE_U1)
        assert np.array_equal(phi[mask], u1[mask]), mode     # the g of a solve is that of its u1
        assert np.abs(phi - ref)[mask].max() <= (DD_TOL if bdd else G_TOL) * top, mode
        assert np.abs(u1 - parts["u1"]).max() <= (G_TOL if mode == "FP64" else DD_TOL) * top, mode
        got[mode, bdd] = phi
    # every length has an FFT: DF32 is FP64
    assert np.array_equal(got["DF32", 0], got["FP64", 0])
