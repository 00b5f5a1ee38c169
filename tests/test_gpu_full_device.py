"""Calls that need no device memory of their own, or can do without the part they lack, on a device
that other arrays fill up."""
import contextlib

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2606_12850_gb300 import build, inputs, sem  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def library():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    return sem.lib()


@contextlib.contextmanager
def full_device(leave=0):
    """Within it, other arrays hold the free device memory but for ``leave`` bytes, to within 4 MB."""
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    held = []
    step = 1 << 38
    while step >= 2 << 20:
        free = torch.cuda.mem_get_info()[0] - leave
        if free < step:
            step >>= 1
            continue
        try:
            held.append(torch.empty(step, dtype=torch.uint8, device="cuda"))
        except torch.OutOfMemoryError:
            step >>= 1
    try:
        yield
    finally:
        held.clear()
        torch.cuda.empty_cache()


def test_gradients_to_the_host():
    w = inputs.layered_cube(5, n=16, side=2000.0, nrec_side=2)  # 4 MB of float64 a gradient
    s = sem.setup_workload(w)
    u = torch.from_numpy(inputs.uniform(5, (5, w.mesh.nglob, 3), -1, 1).astype(np.float32)).cuda()
    G = torch.from_numpy(inputs.uniform(6, (3, len(s.rec_nodes), 3), -1, 1).astype(np.float32)).cuda()
    torch.cuda.synchronize()
    sem.sem_adjoint_begin(s.ctx)
    sem.sem_adjoint_segment(s.ctx, 3, G, u)
    ref = sem.sem_adjoint_gradients(s.ctx)
    with full_device():
        again = sem.sem_adjoint_gradients(s.ctx)
    for a, b in zip(ref, again):
        assert np.any(a != 0.0) and np.array_equal(a, b)
    # the accumulators go on from there: a second segment adds its terms and nothing else
    sem.sem_adjoint_segment(s.ctx, 3, G, u)
    both = sem.sem_adjoint_gradients(s.ctx)
    sem.sem_adjoint_begin(s.ctx)
    sem.sem_adjoint_segment(s.ctx, 3, G, u)
    sem.sem_adjoint_segment(s.ctx, 3, G, u)
    for a, b in zip(sem.sem_adjoint_gradients(s.ctx), both):
        assert np.linalg.norm(a - b) <= 1e-6 * np.linalg.norm(a)


def test_surrogate_without_room_for_the_packed_activations():
    """A max_batch whose general buffers fit and whose packed ones (210 MB beside 1.1 GB here) do not:
    the model is created and the general kernels take its calls."""
    from paper_2606_12850_gb300 import surrogate
    spec = surrogate.Spec()
    flat = spec.init_params(9)
    x = torch.from_numpy(inputs.uniform(10, (3, 9), -1, 1).astype(np.float32)).cuda()
    t = torch.from_numpy(inputs.uniform(11, (3, spec.out_c, spec.out_l), -1, 1).astype(np.float32)).cuda()
    small = surrogate.Spec(in_dim=9, hidden=24, c0=6, l0=7, stage_cout=(10, 8, 12), stage_up=(2, 2, 1), contract=6)
    warm = surrogate.Model(small, max_batch=4)  # loads the general kernels
    warm.set_params(small.init_params(1))
    warm.loss_grad(x, torch.zeros((3, small.out_c, small.out_l), device="cuda"))

    def use(m):
        m.set_params(flat)
        y = torch.zeros((3, spec.out_c, spec.out_l), device="cuda")
        torch.cuda.synchronize()
        m.forward(x, y)
        return m.info()["device_bytes"], m.loss_grad(x, t), y.cpu().numpy().astype(np.float64), m.get_grads()

    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    before = torch.cuda.mem_get_info()[0]
    m = surrogate.Model(spec, max_batch=64)
    need = before - torch.cuda.mem_get_info()[0]
    ref = use(m)
    del m
    keep = torch.zeros((3, spec.out_c, spec.out_l), device="cuda")  # cached for use()
    del keep
    with full_device(leave=need - (120 << 20)):
        got = use(surrogate.Model(spec, max_batch=64))
    assert ref[0] - got[0] > 120 << 20
    assert abs(got[1] - ref[1]) <= 1e-4 * ref[1]
    for a, b in zip(ref[2:], got[2:]):
        assert np.linalg.norm(a - b) <= 2e-3 * np.linalg.norm(a)
