"""When refinement ends: at the first residual that meets rtol; general kinds a pass later within a decade of it."""
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


def _convection(adjoint, n=128, k=2, seed=11, **kw):
    """(u or lambda, residuals, steps) of one convection problem."""
    from paper_2211_07572_gb300.solver import SlabSolver
    p = inputs.convection(n, 16, k, speed=20.0, field_seed=7, velocity_seeds=(8, 9, 10), rhs_seed=seed)
    f = torch.from_numpy(p.f).cuda()
    s = SlabSolver(2, p.n, p.b, p.kind, kappa=p.kappa, beta=p.beta, **kw)
    if adjoint:
        u, _ = s.adjoint(f, allow_noconv=True)
        r = f - s.apply_transpose(u)
        rel, it = (r.norm(dim=1) / f.norm(dim=1)).cpu().numpy(), None
    else:
        u, rel, it = s.solve(f, allow_noconv=True)
    s.close()
    return u, rel, it


@pytest.mark.parametrize("share", [0.05, 0.2, 0.87, 0.99, 1.01])
@pytest.mark.parametrize("adjoint", [False, True])
def test_general_kinds_take_one_more_pass_within_a_decade(adjoint, share):
    """The same with the nonsymmetric kind: one more pass from a tenth of the tolerance on, state and adjoint."""
    u1, rel, _ = _convection(adjoint, max_refine=1)
    best, _, _ = _convection(adjoint, precision="fp64", rtol=1e-13)
    u, got, it = _convection(adjoint, rtol=float(rel.max()) / share)
    err1, err = ((v - best).norm() / best.norm() for v in (u1, u))
    if share < 0.1:
        assert torch.equal(u, u1)
    else:
        assert got.max() < 0.1 * rel.max() and err < 0.1 * err1
    assert it in ((None,) if adjoint else (1,) if share < 0.1 else (2,))


@pytest.mark.parametrize("n,k,seed", [(48, 1, 11), (48, 2, 12), (64, 2, 11), (80, 1, 12), (96, 1, 13), (96, 2, 12), (112, 1, 11)])
def test_the_extra_pass_cannot_lose_the_tolerance(n, k, seed):
    """rtol just above the residual that rounding allows (the second pass reaches it): where the extra pass leaves a larger
    residual, the iterate before it comes back, with its own residual."""
    u2, r2, _ = _convection(False, n, k, seed, max_refine=2, rtol=0.0)
    u3, r3, _ = _convection(False, n, k, seed, max_refine=3, rtol=0.0)
    u, got, it = _convection(False, n, k, seed, rtol=2.0 * float(r2.max()))
    want_u, want_r = (u3, r3) if r3.max() < r2.max() else (u2, r2)
    assert it == 3 and torch.equal(u, want_u) and np.array_equal(got, want_r)
