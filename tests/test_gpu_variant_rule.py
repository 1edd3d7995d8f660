"""Sweep variants chosen by rule, by the caller and by the autotuner: the autotuner
leaves every bit of the state, takes variants that are one kernel as one, and times
on a sample inside a larger mesh."""
import numpy as np
import pytest
import torch

from workloads import ics

pytestmark = pytest.mark.gpu


def _mesh(root, n, levels, seed=3, **kw):
    from paper_1810_01319_gb300 import Mesh, make_desc
    d = make_desc((root,) * 3, n, levels, bc=(0, 1, 0), gamma=5 / 3, **kw)
    mesh = Mesh(d)
    rng = np.random.default_rng(seed)
    for _ in range(levels):
        mesh = Mesh(d, mesh, (rng.random(mesh.n_leaves) < 0.25).astype(np.int8))
    U = ics.blobs(mesh.leaves, (root,) * 3, n, 4, (0.0,) * 3, (1.0,) * 3, 5 / 3, count=6, seed=seed, abc=0.3)
    if kw.get("dual_energy"):
        U = ics.with_internal_energy(U)
    return mesh, U.to(mesh.dtype).cuda().contiguous()


@pytest.mark.parametrize("precision, count", [(4, 24), (8, 2)])
def test_autotuner_keeps_an_unsynchronised_state(precision, count):
    mesh, U = _mesh(2, 8, 1, precision=precision, dual_energy=1)
    U[:, 5] *= 0.5                       # the synchronisation would reset it
    before = U.clone()
    best, ms = mesh.autotune(U)
    assert torch.equal(U, before)
    assert len(ms) == count and all(0 <= v < count for v in best)
    if precision == 4:                   # streaming variants that differ in the register bound alone
        for v, twin in ((8, 6), (11, 10), (20, 18), (23, 22)):
            assert ms[v] == ms[twin]


def test_autotuner_on_more_leaves_than_its_sample():
    mesh, U = _mesh(17, 8, 0, precision=4)           # 4913 leaves
    before = U.clone()
    mesh.autotune(U)
    torch.cuda.synchronize()
    assert torch.equal(U, before)
