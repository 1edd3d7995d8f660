"""A whole step sweeps each row once (its owner also stores it into the
same-level neighbours' ghost rows); the same step over the leaf range
[0, leaves) (cello_hydro_step_part) sweeps every ghost row in place after a
full refresh.  Both give the same interiors bit for bit, from a state whose
ghost layer is NaN: the step reads no ghost cell that it has not written."""
import numpy as np
import pytest
import torch

from workloads import ics

pytestmark = pytest.mark.gpu


def _mesh(root, n, levels, bc, precision, seed, **kw):
    from paper_1810_01319_gb300 import Mesh, make_desc
    hi = tuple(r / max(root) for r in root)
    d = make_desc(root, n, levels, hi=hi, bc=bc, precision=precision, gamma=5 / 3, **kw)
    mesh = Mesh(d)
    rng = np.random.default_rng(seed)
    for _ in range(levels):
        mesh = Mesh(d, mesh, (rng.random(mesh.n_leaves) < 0.25).astype(np.int8))
    U = ics.blobs(mesh.leaves, root, n, 4, (0.0,) * 3, hi, 5 / 3, count=6, seed=seed, abc=0.3)
    if kw.get("dual_energy"):
        U = ics.with_internal_energy(U)
    return mesh, U.to(mesh.dtype).cuda().contiguous()


# roots of one, two and more blocks (a leaf its own neighbour, one neighbour on both sides), every block size
@pytest.mark.parametrize("root, n, levels, bc", [
    ((1, 1, 1), 8, 0, (0, 0, 0)), ((1, 1, 1), 16, 0, (1, 0, 1)), ((2, 1, 3), 8, 1, (0, 1, 0)),
    ((2, 2, 2), 8, 3, (0, 0, 0)), ((3, 2, 2), 16, 2, (1, 1, 1)), ((2, 2, 2), 32, 1, (0, 0, 1)),
])
@pytest.mark.parametrize("precision, variants", [(8, [0, 1, 0]), (4, [0, 2, 3]), (4, [22, 21, 6]), (4, [8, 7, 23])])
def test_whole_step_equals_every_row_in_place(root, n, levels, bc, precision, variants):
    mesh, U = _mesh(root, n, levels, bc, precision, 3)
    mesh.set_sweep_variants(variants)
    _compare(mesh, U, n)


@pytest.mark.parametrize("precision, variants", [(8, [1, 0, 1]), (4, [4, 5, 1]), (4, [11, 20, 9])])
@pytest.mark.parametrize("kw", [dict(riemann=1, steepening=1), dict(dual_energy=1)])
def test_whole_step_of_the_method_variants(precision, variants, kw):
    mesh, U = _mesh((2, 2, 2), 16, 2, (0, 1, 0), precision, 5, **kw)
    mesh.set_sweep_variants(variants)
    _compare(mesh, U, 16)


def _compare(mesh, U, n):
    inner = (slice(None), slice(None)) + (slice(4, 4 + n),) * 3
    dt = torch.zeros(1, dtype=torch.float64, device="cuda")
    mesh.reduce(U, 0.4, dt_next=dt)
    V = torch.full_like(U, float("nan"))
    V[inner] = U[inner]
    for cycle in (0, 1, 2):
        W = V.clone()
        mesh.hydro_step_part(W, dt, cycle, 0, mesh.n_leaves, 0)
        mesh.hydro_step_part(W, dt, cycle, 0, mesh.n_leaves, 1)
        mesh.hydro_step(V, dt, cycle)
        assert torch.isfinite(V[inner]).all()
        assert torch.equal(V[inner], W[inner]), cycle
        fresh = torch.full_like(V, float("nan"))
        fresh[inner] = V[inner]
        V = fresh
