"""Float32 refinement flags of dual-energy states whose pressure comes from a rho e
that is large beside E: one slope within float32's rounding of the threshold on
each leaf, decided as in float64 (exact)."""
import numpy as np
import pytest
import torch

import helpers as H
from oracle import hydro as OH
from oracle import mesh as OM

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("large", [1.0, 1e2, 1e4, 1e8])
@pytest.mark.parametrize("tau", [1e-4, 0.02])
def test_float32_flags_from_a_large_internal_energy(large, tau):
    from paper_1810_01319_gb300 import Mesh
    od = H.oracle_desc(root=(8, 8, 8), n=8, lmax=1, dual_energy=True)
    om = OM.root_mesh(od)
    gm = Mesh(H.gpu_desc(od, 4))
    rng = np.random.default_rng(11)
    U = np.zeros((om.n_leaves, 6, 16, 16, 16), np.float32)
    U[:, 0], U[:, 1], U[:, 4] = 1.0, 1.0, 0.5          # E = kinetic energy: the pressure is that of rho e
    for b in range(om.n_leaves):
        c = np.float32(large * rng.uniform(0.5, 2))
        h = tau * float(c) * (1 + rng.uniform(-3e-4, 3e-4) * min(1.0, 1e-4 / tau))
        U[b, 5] = c
        U[b, 5, 8, 8, 9], U[b, 5, 8, 8, 7] = float(c) + h, float(c) - h
    t = torch.from_numpy(U)
    fo = OH.refine_flags(t.double(), om, 4, tau, tau).numpy()
    assert 0.2 < (fo > 0).mean() < 0.8
    assert np.array_equal(gm.refine_flags(t.cuda().contiguous(), 4, tau, tau).cpu().numpy(), fo)
