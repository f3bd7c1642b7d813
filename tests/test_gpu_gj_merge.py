"""Tournament pivoting with several groups of candidate rows: merges of two to five winner sets, the last group and the last
merge incomplete, one and two levels of merges."""
import numpy as np
import pytest
import torch

from paper_2211_07572_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("n,b", [(576, 32), (832, 32), (1088, 32)])     # 3, 4 and 5 groups in the first panel
def test_first_pass_residual_with_merges(n, b, precision):
    """Relative residual of one pass, state and adjoint.  Rounding leaves eps |A| |u| / |f| with |A| = 8 n^2 and, for a normal load,
    |u| / |f| near 0.05 / n: 0.4 n eps; a hundred times that for the elimination's growth."""
    from paper_2211_07572_gb300.solver import SlabSolver
    p = inputs.convection(n, b, 2, speed=20.0, field_seed=7, velocity_seeds=(8, 9, 10), rhs_seed=11)
    f = torch.from_numpy(p.f).cuda()
    s = SlabSolver(2, n, b, p.kind, kappa=p.kappa, beta=p.beta, precision=precision, max_refine=0)
    _, rel, _ = s.solve(f, allow_noconv=True)
    lam, _ = s.adjoint(f, allow_noconv=True)
    back = ((f - s.apply_transpose(lam)).norm(dim=1) / f.norm(dim=1)).cpu().numpy()
    s.close()
    bound = 40 * n * (2.0 ** -24 if precision == "fp32" else 2.0 ** -53)
    assert rel.max() <= bound and back.max() <= bound
    assert np.isfinite(rel).all()
