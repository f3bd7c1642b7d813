"""What a 2-D factor holds: its coefficients, the slab trees, the interface system and Stage 2's arrays, and no second copy of the
interface columns beside them."""
import numpy as np
import pytest
import torch

from paper_2211_07572_gb300 import inputs

pytestmark = pytest.mark.gpu


def _counts(n, b):
    s, m, slabs = n - 1, b - 1, n // b
    sp = -(-s // 64) * 64
    per_height = slabs * s.bit_length() * m * sp                 # one side, one orientation
    return s, m, slabs, sp * sp, slabs * (s + 1) * m * m, per_height


@pytest.mark.parametrize("n,b", [(256, 32), (300, 12)])
def test_symmetric_factor(n, b):
    from paper_2211_07572_gb300.solver import SlabSolver
    s, m, slabs, blk, node, per_height = _counts(n, b)
    NI = slabs - 1
    want = 8 * (3 * (n + 1) ** 2 + 7 * node + (2 + 4) * per_height + (2 * NI - 1) * blk + (3 * NI + NI + NI - 1) * blk)
    h = SlabSolver(2, n, b, inputs.POISSON, precision="fp64", stage2="sweep")
    got = h.device_bytes
    h.close()
    assert got <= want + want // 100 + 2**20, (got, want)


def test_nonsymmetric_factor():
    """S^-1, S^-T, four m x 2m couplings and R per node; four families of interface columns and the condensed rows in both
    orientations per height; T's three families of blocks, Stage 2's five and the six of the elimination's work."""
    from paper_2211_07572_gb300.solver import SlabSolver
    n, b = 256, 32
    s, m, slabs, blk, node, per_height = _counts(n, b)
    NI = slabs - 1
    p = inputs.convection(n, b, k=1)
    want = 8 * (6 * (n + 1) ** 2 + (2 + 8 + 4) * node + (4 * 2 + 4 + 4) * per_height + (3 * NI + 5 * (NI - 1) + 6) * blk)
    h = SlabSolver(2, n, b, inputs.CONVECTION, kappa=p.kappa, beta=p.beta, precision="fp64")
    got = h.device_bytes
    u, rel, _ = h.solve(torch.from_numpy(p.f).cuda())
    lam, _ = h.adjoint(u, u)
    back = h.apply_transpose(lam)
    h.close()
    assert got <= want + want // 100 + 2**20, (got, want)
    assert rel.max() <= 1e-10
    assert float((back - u).norm() / u.norm()) <= 1e-9
