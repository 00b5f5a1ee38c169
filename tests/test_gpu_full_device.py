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
