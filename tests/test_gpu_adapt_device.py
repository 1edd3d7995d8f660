"""Mesh adaptation on the device against the oracle: random refine/coarsen
sequences on root arrays of one and more blocks (leaves, neighbour table, remap,
all exact), float32 refinement flags decided in float32 or float64 (exact, with
states that sit on and next to the thresholds), and the remap's refusal."""
import numpy as np
import pytest
import torch

import helpers as H
from oracle import hydro as OH
from oracle import mesh as OM

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("root, lmax, bc", [((1, 1, 1), 4, (0, 0, 0)), ((1, 1, 1), 3, (1, 0, 1)),
                                            ((2, 1, 3), 3, (0, 1, 0)), ((3, 2, 2), 2, (1, 1, 1)),
                                            ((2, 2, 2), 4, (0, 0, 0))])
@pytest.mark.parametrize("precision", [4, 8])
def test_random_adaptations(root, lmax, bc, precision):
    from paper_1810_01319_gb300 import Mesh
    od = H.oracle_desc(root=root, n=8, lmax=lmax, bc=bc)
    d = H.gpu_desc(od, precision)
    om, gm = OM.root_mesh(od), Mesh(d)
    rng = np.random.default_rng(sum(root) * 10 + lmax)
    for step in range(7):
        p = (0.05, 0.6, 0.35) if step < 3 else (0.75, 0.2, 0.05)     # grow, then coarsen
        f = rng.choice([-1, 0, 1], size=om.n_leaves, p=p).astype(np.int8)
        om2, gm2 = OM.build(od, om, f), Mesh(d, gm, f)
        assert np.array_equal(gm2.leaves.astype(np.int64), om2.leaves), step
        kind, idx, fine8 = gm2.neighbour_table()
        ok, oi, of = OM.neighbour_table(om2)
        assert np.array_equal(kind, ok) and np.array_equal(idx, oi) and np.array_equal(fine8, of)
        g = torch.Generator().manual_seed(step)
        U = torch.rand(om.n_leaves, 5, 16, 16, 16, generator=g, dtype=torch.float64) + 0.5
        U = U.to(gm.dtype)
        Ug = U.cuda().contiguous()
        gm.ghost_refresh(Ug)
        if precision == 8:
            Uo = OH.remap(OH.ghost_refresh(U, om), om, om2)
            assert torch.equal(H.interior(gm2.remap_from(gm, Ug).cpu(), 8), H.interior(Uo, 8))
        om, gm = om2, gm2
        if om.n_leaves > 400:
            break


def test_remap_refuses_unrelated_meshes():
    from paper_1810_01319_gb300 import CelloError, Mesh
    od = H.oracle_desc(root=(1, 1, 1), n=8, lmax=2)
    d = H.gpu_desc(od, 8)
    fine = Mesh(d, Mesh(d), np.ones(1, np.int8))
    fine = Mesh(d, fine, np.ones(8, np.int8))
    U = fine.empty_state().normal_()
    coarse = Mesh(d)                       # two levels coarser everywhere: no children one level finer
    V = torch.full((1, 5, 16, 16, 16), 3.0, dtype=torch.float64, device="cuda")
    with pytest.raises(CelloError, match="one adaptation apart"):
        coarse.remap_from(fine, U, V)
    assert bool((V == 3.0).all())


def test_remap_from_several_threads():
    """Two old meshes and two states each, remapped into one new mesh at the same time."""
    import threading
    from paper_1810_01319_gb300 import Mesh
    od = H.oracle_desc(root=(3, 2, 2), n=8, lmax=2)
    d = H.gpu_desc(od, 8)
    root = Mesh(d)
    neu = Mesh(d, root, np.array([1] * 3 + [0] * 9, np.int8))
    jobs = []
    for old in (root, Mesh(d, neu, np.ones(neu.n_leaves, np.int8))):
        for k in range(2):
            U = torch.rand(old.n_leaves, 5, 16, 16, 16, dtype=torch.float64, device="cuda") + 0.5
            old.ghost_refresh(U)
            jobs.append((old, U, neu.remap_from(old, U), torch.zeros_like(neu.empty_state()), torch.cuda.Stream()))
    torch.cuda.synchronize()

    def work(old, U, want, got, stream):
        for _ in range(50):
            neu.remap_from(old, U, got, stream=stream)

    threads = [threading.Thread(target=work, args=j) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    for old, U, want, got, stream in jobs:
        assert torch.equal(got, want)


def test_neighbour_table_during_a_capture():
    from paper_1810_01319_gb300 import Mesh
    od = H.oracle_desc(root=(2, 2, 1), n=8, lmax=1)
    gm = Mesh(H.gpu_desc(od, 8))
    want = gm.neighbour_table()
    x, g = torch.zeros(4, device="cuda"), torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        x += 1
        got = gm.neighbour_table()
        x += 1
    g.replay()
    torch.cuda.synchronize()
    assert all(np.array_equal(a, b) for a, b in zip(got, want)) and bool((x == 2).all())


@pytest.mark.parametrize("dual", [False, True])
@pytest.mark.parametrize("field", [0, 4])
@pytest.mark.parametrize("tau, tau_c", [(0.3, 0.075), (0.3, 0.3), (0.0, 0.0), (1e-30, 1e-30), (0.25, -0.5)])
def test_float32_flags_on_the_thresholds(dual, field, tau, tau_c):
    from paper_1810_01319_gb300 import Mesh
    od = H.oracle_desc(root=(3, 2, 2), n=8, lmax=2, dual_energy=dual)
    om = OM.build(od, OM.root_mesh(od), np.array([1, 0, 0, 0, 0, 0, 0, 1, 0, 0, 0, 0], np.int8))
    gm = Mesh(H.gpu_desc(od, 4), leaves=om.leaves)
    B = om.n_leaves
    rng = np.random.default_rng(7)
    U = np.zeros((B, 6 if dual else 5, 16, 16, 16), np.float32)
    for b in range(B):      # leaf by leaf: a slope just below, at and just above each threshold, noise, floors
        rho = np.ones((16, 16, 16), np.float32)
        kindb = b % 8
        if kindb < 5:
            jump = np.float32(2 * abs((tau, tau_c)[b % 2]))
            for _ in range(abs(kindb - 2)):
                jump = np.nextafter(jump, np.float32(0 if kindb < 2 else 9))
            rho[8, 8, 8] = np.float32(1) + jump
        elif kindb == 5:
            rho += rng.uniform(0, 0.2, rho.shape).astype(np.float32)
        elif kindb == 6:
            rho[5, 5, 5] = 1e-12
        U[b, 0] = rho
        U[b, 1] = rng.normal(0, 0.1 * (b % 3), rho.shape).astype(np.float32)
        E = 1.5 * (rho if field == 4 else 1.0) + 0.5 * U[b, 1] ** 2 / np.maximum(rho, 1e-6)
        U[b, 4] = E.astype(np.float32)
        if dual:
            U[b, 4] *= 1.0 if b % 2 else 300.0
            U[b, 1] *= 1.0 if b % 2 else 24.0
            U[b, 5] = np.float32(1.5) * rho
    t = torch.from_numpy(U)
    fo = OH.refine_flags(t.double(), om, field, tau, tau_c).numpy()
    fg = gm.refine_flags(t.cuda().contiguous(), field, tau, tau_c).cpu().numpy()
    assert np.array_equal(fg, fo)
