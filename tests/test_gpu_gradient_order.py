"""The adjoint's gradients on the device (float32, caller order) equal the host ones rounded, bit
for bit, on meshes whose sweep order is not the caller's, at orders with and without padded
workspaces; arrays left out are skipped."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2606_12850_gb300 import build, inputs, sem  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ngll,n", [(2, 5), (4, 3), (5, 3), (8, 2)])
def test_device_gradients_equal_host_ones(ngll, n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    w = inputs.layered_cube(ngll, n=n, side=600.0, nrec_side=2)
    s = sem.setup_workload(w)
    N = 14  # a graph of ten adjoint steps, then single ones
    u = torch.from_numpy(inputs.uniform(5, (N + 2, w.mesh.nglob, 3), -1, 1).astype(np.float32)).cuda()
    G = torch.from_numpy(inputs.uniform(6, (N, len(s.rec_nodes), 3), -1, 1).astype(np.float32)).cuda()
    torch.cuda.synchronize()
    sem.sem_adjoint_begin(s.ctx)
    sem.sem_adjoint_segment(s.ctx, N, G, u)
    host = sem.sem_adjoint_gradients(s.ctx)
    dev = [torch.full((w.mesh.nspec, ngll ** 3), float("nan"), device="cuda") for _ in range(3)]
    torch.cuda.synchronize()
    sem.sem_adjoint_gradients_dev(s.ctx, dev[0], None, dev[2])
    sem.sem_adjoint_gradients_dev(s.ctx, None, dev[1], None)
    sem.sem_sync(s.ctx)
    for h, d in zip(host, dev):
        assert np.any(h != 0.0)
        assert np.array_equal(h.astype(np.float32), d.cpu().numpy())
