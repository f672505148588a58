"""Device memory of a plan (GPU)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# bytes of a 3-D plan whose boundary spectra are kept in one form (FP64), for each axis, with
# the temporaries that made them
ONE_FORM = {(129, 129, 129): 457.9e6, (257, 193, 129): 1276.7e6, (257, 257, 257): 2883.5e6}


@pytest.mark.parametrize("n", list(ONE_FORM), ids=lambda n: "x".join(map(str, n)))
def test_a_plan_takes_no_more_than_one_form_of_the_spectra(n):
    import paper_2108_11871_gb300 as idp
    plan = idp.create_plan(3, n, [1.0 / (max(n) - 1)] * 3, 6)
    assert idp.plan_info(plan)["workspace_bytes"] <= ONE_FORM[n]
    idp.plan_check_guards(plan)


@pytest.mark.parametrize("h", [(1.0, 1.0, 1.0), (2.0, 1.0, 1.0), (1.0, 2.0, 3.0)], ids=["equal", "two_equal", "unequal"])
def test_axes_share_spectra_only_where_they_are_the_same(h):
    import torch
    import workloads as w
    from oracle import greens as ogreens
    import paper_2108_11871_gb300 as idp
    n = (33, 33, 33)
    h = [v / 32.0 for v in h]
    rho = w.random_interior(n, seed=2)
    ref = ogreens.boundary_convolution(rho, h)
    r = torch.from_numpy(rho).cuda()
    out = torch.empty_like(r)
    mask = ogreens.boundary_mask(n)
    # FP64 spectra, their fixed-point form, and the double-float form
    for precision, bdd, tol in ((idp.IDP_PRECISION_FP64, 0, 1e-14), (idp.IDP_PRECISION_MIXED_BF16X3, 0, 1e-14),
                                (idp.IDP_PRECISION_MIXED_BF16X3, 1, 1e-12)):
        plan = idp.create_plan(3, n, h, 4)
        idp.plan_set(plan, idp.IDP_KEY_PRECISION, precision)
        idp.plan_set(plan, idp.IDP_KEY_MIXED_BOUNDARY_DF32, bdd)
        idp.solve(plan, r, out)
        torch.cuda.synchronize()
        idp.plan_status(plan)
        assert np.abs(out.cpu().numpy() - ref)[mask].max() <= tol * np.abs(ref[mask]).max()
