"""Meshes whose sizes differ by orders of magnitude between the axes (GPU).  The transformed layers of
gtilde and of E scale like 1 / h_s^2 and are summed on one unit in the expansions, so that the
weakest axis keeps the fewest bits.  u1, against the oracle: both err by a few 1e-14 here, the
FP64 layers' error too (against 80-bit references at 129^2, largest error of u1 in FP64 and now:
mesh ratio 1 4.5e-15 and 1.0e-15, 100 1.8e-14 and 2.0e-14, 1e4 1.6e-14 and 1.6e-14)."""
import numpy as np
import pytest

from oracle import solve as osolve

pytestmark = pytest.mark.gpu

CASES = [((129, 129), (1.0, 100.0)), ((129, 129), (1e4, 1.0)), ((65, 33, 65), (1.0, 30.0, 1000.0)),
         ((33, 65, 33), (1e4, 1.0, 1e4))]


@pytest.mark.parametrize("n,h", CASES, ids=["x".join(map(str, n)) + "_%g" % max(h) for n, h in CASES])
def test_stretched_mesh(n, h):
    import torch
    import paper_2108_11871_gb300 as idp
    h = [v / 128.0 for v in h]
    x = np.meshgrid(*[np.linspace(-1.0, 1.0, k) for k in n], indexing="ij")
    rho = np.maximum(0.0, 1.0 - sum(c * c for c in x) / 0.64) ** 8 * (1.0 + 0.3 * np.sin(9.0 * x[0] + 2.0 * x[1]))
    parts = {}
    phi = osolve.solve(rho, h, 6, boundary="convolution", parts=parts)
    plan = idp.create_plan(len(n), n, h, 6)
    r = torch.from_numpy(rho).cuda()
    out = torch.empty_like(r)
    for stage, ref in ((idp.IDP_STAGE_U1, parts["u1"]), (idp.IDP_STAGE_PHI, phi)):
        idp.solve_stage(plan, stage, r, out)
        torch.cuda.synchronize()
        assert np.abs(out.cpu().numpy() - ref).max() <= 2e-13 * np.abs(ref).max()
