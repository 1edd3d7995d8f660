"""Tracers that are not inside the leaf they name (NaN and infinite positions, far
outside the box, another leaf's index) among ordinary ones: the ordinary ones move
as without them, the others keep a leaf index of the mesh or are lost."""
import numpy as np
import pytest
import torch

from workloads import ics

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [4, 8])
@pytest.mark.parametrize("bc", [(0, 0, 0), (1, 0, 1)])
def test_tracers_outside_their_leaf(precision, bc):
    from paper_1810_01319_gb300 import Mesh, make_desc
    d = make_desc((2, 2, 2), 8, 1, bc=bc, precision=precision, gamma=5 / 3)
    mesh = Mesh(d, Mesh(d), np.array([1, 0, 0, 1, 0, 0, 0, 0], np.int8))
    U = ics.blobs(mesh.leaves, (2,) * 3, 8, 4, (0.0,) * 3, (1.0,) * 3, 5 / 3, count=4, seed=1, abc=0.3)
    U = U.to(mesh.dtype).cuda().contiguous()
    mesh.ghost_refresh(U)
    P = 3000
    pos = torch.rand(3, P, generator=torch.Generator().manual_seed(2), dtype=torch.float64).cuda()
    leaf = mesh.particles_locate(pos)
    dt = torch.full((1,), 1e-2, dtype=torch.float64, device="cuda")
    want_pos, want_leaf = pos.clone(), leaf.clone()
    mesh.particles_push(U, want_pos, want_leaf, dt)
    sick = torch.zeros(P, dtype=torch.bool)
    bad = [float("nan"), float("inf"), -float("inf"), 1e300, -1e300, 7.5, -3.25, 2.0 ** 31, -2.0 ** 40]
    for k, v in enumerate(bad):
        for a in range(3):
            i = 100 * k + 10 * a
            sick[i] = True
            pos[a, i] = v
    for i in range(2000, 2050):                        # the index of another leaf
        sick[i] = True
        leaf[i] = (leaf[i] + 5) % mesh.n_leaves
    for step in range(2):
        mesh.particles_push(U, pos, leaf, dt)
        assert bool(((leaf >= -1) & (leaf < mesh.n_leaves)).all())
        if step == 0:
            ok = ~sick.cuda()
            assert torch.equal(pos[:, ok], want_pos[:, ok]) and torch.equal(leaf[ok], want_leaf[ok])
