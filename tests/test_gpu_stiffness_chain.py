"""f = -K u applied to its own result, call after call without a wait in between (a power iteration,
a Krylov method): each call's kernels start while the call before still writes the array they read.
Equal, bit for bit, to the same calls with a wait after each; patch sweep and element kernel, caller
arrays and the solver's layout."""
import pytest

torch = pytest.importorskip("torch")

from paper_2606_12850_gb300 import build, inputs, sem  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("stride", [3, 4])
@pytest.mark.parametrize("assembly", [0, 1])
@pytest.mark.parametrize("ngll,n", [(3, 24), (5, 16), (8, 7)])
def test_back_to_back_applications(ngll, n, assembly, stride):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    mesh = inputs.structured_hex_mesh(n, ngll, 1.0, jitter=0.1, seed=3)  # unit moduli: values stay of order one
    one = inputs.uniform(2, mesh.ibool.shape, 0.9, 1.1)
    ctx = sem.sem_create(ngll, 0)
    sem.sem_set_option(ctx, sem.SEM_OPT_ASSEMBLY, assembly)
    sem.sem_set_mesh_corners(ctx, mesh.ibool, mesh.ctrl, mesh.nglob)
    sem.sem_set_material(ctx, one, 1.5 * one, 0.8 * one)
    first = torch.zeros((mesh.nglob, stride), device="cuda")
    first[:, :3] = torch.from_numpy(inputs.random_field(mesh.nglob, 6)).cuda()
    out = []
    for wait in (True, False):
        a, b = first.clone(), torch.zeros_like(first)
        torch.cuda.synchronize()
        for k in range(12):
            if stride == 3:
                sem.sem_apply_stiffness(ctx, a, b)
            else:
                sem.sem_apply_stiffness_strided(ctx, a, b, 4)
            if wait:
                sem.sem_sync(ctx)
            a, b = b, a
        sem.sem_sync(ctx)
        out.append(a)
    assert bool(torch.isfinite(out[0]).all()) and bool((out[0][:, :3] != 0).any())
    assert torch.equal(out[0], out[1])
