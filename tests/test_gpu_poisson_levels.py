"""The multigrid solver over the level structures it chooses between: block
levels of every edge, periodic arrays on tiles (edge a multiple of 4), on the
single-array kernels and in the one-CTA bottom, odd coarsest grids, one block
that is its own neighbour.  float64: the oracle's cycles, whose only difference
is the order of the two mean removals (the bound of the other mg0 tests, 1e-12
of the largest value).  Mixed precision: 14 cycles reach the float64 solution of
14 cycles to 1e-6 of the largest value (each cycle contracts the error by 4 at
least: 4^-14 = 4e-9 of it is left on either side)."""
import numpy as np
import pytest
import torch

import helpers as H
from oracle import mesh as OM
from oracle import poisson as OP

pytestmark = pytest.mark.gpu


def _solve(root, n, level, cycles, inner, seed):
    od = H.oracle_desc(root=(root,) * 3, n=n, lmax=level)
    om = OM.root_mesh(od)
    flags = []
    for _ in range(level):
        f = np.ones(om.n_leaves, dtype=np.int8)
        om = OM.build(od, om, f)
        flags.append(f)
    gm = H.gpu_mesh_from_flags(od, flags, 8)
    g = torch.Generator().manual_seed(seed)
    f = torch.randn(om.n_leaves, n, n, n, generator=g, dtype=torch.float64) + 0.25
    phi, res = gm.poisson_solve(f.cuda().contiguous(), cycles, inner=inner)
    quiet, _ = gm.poisson_solve(f.cuda().contiguous(), cycles, inner=inner, residuals=False)
    assert torch.equal(phi, quiet)
    po, ro = OP.solve(OP.to_global(om, f), od.dx(level), cycles)
    return phi.cpu(), res, OP.from_global(om, po), ro


# arrays below the blocks: 2, 4, 6, 10, 14 (-> 7), 2 x 4 = 8 -> 16, 24, 28 cells per edge
@pytest.mark.parametrize("root,n,level", [(1, 8, 0), (1, 32, 0), (2, 8, 0), (3, 8, 0), (5, 8, 0), (7, 8, 0),
                                          (2, 8, 2), (6, 8, 1), (7, 8, 1), (2, 32, 0)])
def test_float64_cycles_match_the_oracle(root, n, level):
    phi, res, expect, ro = _solve(root, n, level, 3, 8, root * 100 + n)
    assert float((phi - expect).abs().max()) <= 1e-12 * float(expect.abs().max())
    assert np.allclose(res, ro, rtol=1e-6, atol=0)


@pytest.mark.parametrize("root,n,level", [(1, 8, 0), (3, 8, 0), (9, 8, 0), (2, 16, 1), (5, 8, 1), (4, 32, 0)])
def test_mixed_cycles_reach_the_solution(root, n, level):
    phi, res, expect, ro = _solve(root, n, level, 14, 4, root * 100 + n)
    assert float((phi - expect).abs().max()) <= 1e-6 * float(expect.abs().max())
    assert np.allclose(res[:5], ro[:5], rtol=1e-3, atol=0)
