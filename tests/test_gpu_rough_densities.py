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
    plan = idp.create_plan(len(n), n, h, 4)
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
