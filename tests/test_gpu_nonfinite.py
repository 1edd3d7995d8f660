"""One cell that is not finite, one step.  In a supersonic stream the cell stays so
and the reduction reports it, and every cell beyond the sweeps' stencil (four cells
along each axis) has the bits of the step without it."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("riemann, steepening", [(0, 0), (1, 0), (1, 1)])
@pytest.mark.parametrize("precision, variant", [(4, 0), (4, 6), (4, 22), (8, 1)])
@pytest.mark.parametrize("field, value", [(1, float("nan")), (2, float("nan")), (4, float("nan")), (1, float("inf"))])
def test_sick_cell_in_a_supersonic_stream(field, value, precision, variant, riemann, steepening):
    from paper_1810_01319_gb300 import CelloError, Mesh, make_desc
    n, root = 16, 2
    mesh = Mesh(make_desc((root,) * 3, n, 0, precision=precision, gamma=5 / 3, riemann=riemann, steepening=steepening))
    mesh.set_sweep_variant(variant)
    g = torch.Generator().manual_seed(5)
    U = mesh.empty_state(device="cpu").zero_()
    U[:, 0] = 1 + 0.01 * torch.rand(U[:, 0].shape, generator=g)
    for q, u in ((1, 6.0), (2, -6.0), (3, 0.3)):            # sound speed 1.3
        U[:, q] = u * U[:, 0]
    U[:, 4] = 1.5 + 0.5 * (U[:, 1] ** 2 + U[:, 2] ** 2 + U[:, 3] ** 2) / U[:, 0]
    U = U.cuda().contiguous()
    dt = torch.zeros(1, dtype=torch.float64, device="cuda")
    mesh.reduce(U, 0.4, dt_next=dt)
    mesh.check()
    leaf, at = 0, (4 + 7, 4 + 9, 4 + 5)                     # z, y, x
    V = U.clone()
    V[(leaf, field) + at] = value
    mesh.hydro_step(U, dt, 0)
    mesh.hydro_step(V, dt, 0)
    assert not torch.isfinite(V[(leaf, slice(None)) + at]).all()
    mesh.reduce(V, 0.4, dt_next=torch.zeros_like(dt))
    with pytest.raises(CelloError):
        mesh.check()
    differs = torch.zeros(mesh.n_leaves, n, n, n, dtype=torch.bool)
    cells = slice(4, 4 + n)
    for a, b in zip(U.cpu().unbind(1), V.cpu().unbind(1)):
        a, b = a[:, cells, cells, cells], b[:, cells, cells, cells]
        differs |= a != b
    N = n * root
    lv = mesh.leaves
    for b in range(mesh.n_leaves):
        x, y, z = (np.arange(n) + int(lv[b, 1 + a]) * n for a in range(3))
        far = [np.minimum((c - s) % N, (s - c) % N) > 4 for c, s in ((z, 7), (y, 9), (x, 5))]
        out = torch.from_numpy(far[0][:, None, None] | far[1][None, :, None] | far[2][None, None, :])
        assert not differs[b][out].any(), b


@pytest.mark.parametrize("variant", [0, 6, 22])
@pytest.mark.parametrize("field", [1, 2, 3])
def test_slope_beside_a_nan_is_that_of_float64(field, variant):
    """Slow flow with jumps of the order of the values from cell to cell: the cells that
    stay finite beside a NaN are those of the float64 step to the float32 bar (2e-5 of
    the largest value); a slope that is not 0 beside it moves them by percents."""
    from paper_1810_01319_gb300 import Mesh, make_desc
    n, out, dt = 16, [], None
    for precision in (8, 4):
        mesh = Mesh(make_desc((1, 1, 1), n, 0, precision=precision, gamma=5 / 3))
        mesh.set_sweep_variant(variant if precision == 4 else 0)
        g = torch.Generator().manual_seed(9)
        U = mesh.empty_state(device="cpu").zero_()
        U[:, 0] = 1 + 0.2 * torch.rand(U[:, 0].shape, generator=g)
        for q in (1, 2, 3):
            U[:, q] = 0.3 * torch.randn(U[:, 0].shape, generator=g) * U[:, 0]
        U[:, 4] = 1.5 + 0.5 * (U[:, 1] ** 2 + U[:, 2] ** 2 + U[:, 3] ** 2) / U[:, 0]
        U = U.float().to(mesh.dtype).cuda().contiguous()
        if dt is None:
            dt = torch.zeros(1, dtype=torch.float64, device="cuda")
            mesh.reduce(U, 0.2, dt_next=dt)
        U[0, field, 11, 12, 10] = float("nan")
        mesh.hydro_step(U, dt, 0)
        out.append(U[0, :, 4:4 + n, 4:4 + n, 4:4 + n].double().cpu())
    both = torch.isfinite(out[0]) & torch.isfinite(out[1])
    assert both.float().mean() > 0.5 and not both.all()
    assert float((out[0] - out[1])[both].abs().max()) <= 2e-5 * float(out[0][both].abs().max())
