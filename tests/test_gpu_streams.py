"""Two states of one mesh stepped on two streams at the same time: with one
level and no reduction asked for, the steps share nothing but the mesh's tables,
and each state equals its own steps in sequence bit for bit; so does a step alone
on the mesh afterwards.  Variants chosen by rule and set, more work items than the
device holds at once, sweeps of unlike item counts beside each other (the cycles'
parities differ, one axis outflows), batched and replayed from graphs."""
import pytest
import torch

from workloads import ics

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("root, n, precision, variants", [
    (4, 16, 4, None), (5, 32, 4, None), (4, 16, 8, None), (6, 8, 4, [14, 21, 17]), (5, 32, 4, [22, 18, 21]),
    (4, 16, 4, [0, 6, 10]),
])
def test_two_states_on_two_streams(root, n, precision, variants, graph):
    from paper_1810_01319_gb300 import EXEC_GRAPH, Mesh, make_desc
    d = make_desc((root,) * 3, n, 0, bc=(0, 1, 0), precision=precision, gamma=5 / 3)
    mesh = Mesh(d)
    if variants:
        mesh.set_sweep_variants(variants)
    U = [ics.blobs(mesh.leaves, (root,) * 3, n, 4, (0.0,) * 3, (1.0,) * 3, 5 / 3, count=6, seed=s, abc=0.3)
         .to(mesh.dtype).cuda().contiguous() for s in (1, 2)]
    inner = (slice(None), slice(None)) + (slice(4, 4 + n),) * 3
    dt = torch.zeros(1, dtype=torch.float64, device="cuda")
    mesh.reduce(U[0], 0.1, dt_next=dt)
    want = [u.clone() for u in U]
    steps = 50
    for k in range(2):
        for c in range(steps + 1):
            mesh.hydro_step(want[k], dt, c + k)
    if graph:
        mesh.set_exec(EXEC_GRAPH)
    streams = [torch.cuda.Stream() for _ in range(2)]
    torch.cuda.synchronize()
    for c in range(steps):
        for k in range(2):
            mesh.hydro_step(U[k], dt, c + k, stream=streams[k])
    torch.cuda.synchronize()
    for k in range(2):
        mesh.hydro_step(U[k], dt, steps + k)
        assert torch.equal(U[k][inner], want[k][inner])
    mesh.check()
