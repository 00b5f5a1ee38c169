"""The largest shot counts: nodes times shots just below 2^31, where an odd count's padded field
(the shots are kept in pairs) reaches 2^31 slots."""
import pytest

torch = pytest.importorskip("torch")

from paper_2606_12850_gb300 import build, inputs, sem  # noqa: E402

pytestmark = pytest.mark.gpu


def test_nonfinite_value_found_in_the_largest_field():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    shots = 2 ** 28 - 1  # of 8 nodes; three fields of 34 GB and the caller's 26 GB
    if torch.cuda.mem_get_info()[0] < 150e9:
        pytest.skip("needs 150 GB of free device memory")
    mesh = inputs.structured_hex_mesh(1, 2, 100.0)
    ctx = sem.sem_create(2, 0)
    sem.sem_set_mesh_corners(ctx, mesh.ibool, mesh.ctrl, mesh.nglob)
    ones = inputs.uniform(1, mesh.ibool.shape, 1.0, 1.1)
    sem.sem_set_material(ctx, 2500 * ones, 3000 * ones, 1700 * ones)
    sem.sem_set_dt(ctx, 1e-4)
    sem.sem_set_shots(ctx, shots)
    u = torch.zeros(3 * 8 * shots, device="cuda")
    torch.cuda.synchronize()
    sem.sem_set_state_dev(ctx, u)
    sem.sem_check_finite(ctx)
    for at in (0, u.numel() // 2, u.numel() - 1):
        u[at] = float("nan")
        torch.cuda.synchronize()
        sem.sem_set_state_dev(ctx, u)
        with pytest.raises(sem.SemError, match="non-finite"):
            sem.sem_check_finite(ctx)
        u[at] = 0.0
    del ctx, u
    torch.cuda.empty_cache()
