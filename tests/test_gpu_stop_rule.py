"""When refinement ends: at the first residual that meets rtol."""
import numpy as np
import pytest
import torch

from paper_2211_07572_gb300 import inputs

pytestmark = pytest.mark.gpu


def _problem(dim):
    return (inputs.diffusion(35, 7, k=3, dim=3, n_modes=8, field_seed=4, rhs_seed=104) if dim == 3 else
            inputs.diffusion(256, 16, k=2, n_modes=8, field_seed=4, rhs_seed=104))


@pytest.mark.parametrize("share", [0.2, 0.87, 0.88, 0.99, 1.01])
@pytest.mark.parametrize("dim", [2, 3])
def test_symmetric_kinds_end_at_the_tolerance(dim, share):
    """rtol placed so that the residual after one pass is `share` of it: below 1 nothing more runs, above one more pass."""
    from paper_2211_07572_gb300.solver import SlabSolver
    p = _problem(dim)
    f = torch.from_numpy(p.f).cuda()
    kw = dict(kappa=p.kappa, precision="fp32")
    s = SlabSolver(dim, p.n, p.b, p.kind, max_refine=1, rtol=1e-10, **kw)
    u1, rel, _ = s.solve(f, allow_noconv=True)
    s.close()
    s = SlabSolver(dim, p.n, p.b, p.kind, rtol=float(rel.max()) / share, **kw)
    u, got, it = s.solve(f)
    s.close()
    if share < 1:
        assert it == 1 and torch.equal(u, u1) and np.array_equal(got, rel)
    else:
        assert it == 2 and got.max() < 0.1 * rel.max()
