"""Sweep variants chosen by rule, by the caller and by the autotuner: -1 gives a
mesh its rule back; the autotuner leaves every bit of the state, takes variants that
are one kernel as one, and times them on a sample inside a larger mesh; and leaf
ranges whose size makes the rule take the shared-memory form give the bits of whole
steps in the streaming form."""
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


def test_rule_given_back():
    from paper_1810_01319_gb300 import CelloError
    mesh, U = _mesh(2, 16, 0, precision=4)
    dt = torch.zeros(1, dtype=torch.float64, device="cuda")
    mesh.reduce(U, 0.4, dt_next=dt)
    want = U.clone()
    mesh.hydro_step(want, dt, 0)
    mesh.set_sweep_variants([3, 21, 7])
    mesh.set_sweep_variant(-1)
    mesh.set_sweep_variants([-1, 20, -1])
    for bad in ([-2, 0, 0], [0, 24, 0]):
        with pytest.raises(CelloError):
            mesh.set_sweep_variants(bad)
    mesh.hydro_step(U, dt, 0)
    assert torch.equal(U, want)


@pytest.mark.parametrize("kw", [{}, dict(riemann=1, steepening=1), dict(dual_energy=1)])
def test_small_ranges_equal_the_whole_step(kw):
    mesh, V = _mesh(4, 32, 1, precision=4, **kw)     # the whole: 70,000 pencils and more; a range of 8 leaves: 12,800
    dt = torch.zeros(1, dtype=torch.float64, device="cuda")
    mesh.reduce(V, 0.4, dt_next=dt)
    inner = (slice(None),) + (slice(4, 36),) * 3
    for cycle in (0, 1):
        parts = [(b, min(8, mesh.n_leaves - b)) for b in range(0, mesh.n_leaves, 8)]
        want = V.clone()
        mesh.hydro_step(want, dt, cycle)
        pools = [V.clone() for _ in parts]
        for part in (0, 1):                          # every range's face fluxes before any correction
            for W, (b, nb) in zip(pools, parts):
                mesh.hydro_step_part(W, dt, cycle, b, nb, part)
        for W, (b, nb) in zip(pools, parts):
            for leaf in range(b, b + nb):
                assert torch.equal(W[leaf][inner], want[leaf][inner]), (cycle, leaf)
        V = want
