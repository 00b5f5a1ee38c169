"""The rim pass where there is little or nothing else: bricks of one element at NGLL 2 (every node
but the mesh's own corners is shared) and periodic meshes (every node is), against the FP64 oracle.
Bars of the solver: wavefield 2e-5, seismogram 1e-4 relative L2; f = -K u 1e-5."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2606_12850_gb300 import build, inputs, sem  # noqa: E402

pytestmark = pytest.mark.gpu


def rel_l2(a, b):
    return float(np.linalg.norm(np.asarray(a, np.float64) - b) / np.linalg.norm(b))


@pytest.mark.parametrize("dims,periodic", [((4, 3, 5), False), ((4, 4, 4), True), ((2, 3, 4), True)])
@pytest.mark.parametrize("shots", [1, 2, 3])
def test_meshes_of_rim_nodes(oracle, dims, periodic, shots):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    mesh = inputs.structured_hex_mesh(dims, 2, 600.0, periodic=periodic)
    rho, vp = (inputs.uniform(2, mesh.ibool.shape, lo, hi, stream=s) for s, (lo, hi) in
               enumerate(((2200, 2800), (3000, 4000))))
    m = oracle.Model(mesh.ibool, mesh.ctrl, mesh.nglob, rho, vp, vp / 1.8, 2)
    dt = m.cfl_dt(0.3)
    ctx = sem.sem_create(2, 0)
    sem.sem_set_option(ctx, sem.SEM_OPT_PATCH_SHAPE, sem.patch_shape_code(1, 1, 1))
    sem.sem_set_mesh_corners(ctx, mesh.ibool, mesh.ctrl, mesh.nglob)
    sem.sem_set_material(ctx, rho, vp, vp / 1.8)
    sem.sem_set_dt(ctx, dt)
    u = inputs.random_field(mesh.nglob, 6)
    f = torch.full((mesh.nglob, 3), float("nan"), device="cuda")
    ud = torch.from_numpy(u).cuda()
    torch.cuda.synchronize()
    sem.sem_apply_stiffness(ctx, ud, f)
    sem.sem_sync(ctx)
    assert rel_l2(f.cpu().numpy(), m.forces(u.astype(np.float64))) <= 1e-5
    nodes = np.arange(0, mesh.nglob, 3, dtype=np.int32)
    force = inputs.uniform(4, (len(nodes), 3), -1e10, 1e10)
    rec = np.arange(mesh.nglob, dtype=np.int32)
    sem.sem_set_shots(ctx, shots)
    sem.sem_set_shot_sources(ctx, np.arange(len(nodes)) % shots, nodes, force, 20.0, 3.0 * dt)
    sem.sem_set_receiver_nodes(ctx, rec)
    sem.sem_set_state(ctx)
    seis = sem.sem_run(ctx, 13).reshape(shots, len(rec), 3, 13)
    uu = sem.sem_get_state(ctx, want=(True, False, False))[0].reshape(shots, -1, 3)
    for q in range(shots):
        mine = np.arange(len(nodes)) % shots == q
        ref_seis, ref_u, _, _ = oracle.newmark_run(m, dt, 13, src_nodes=nodes[mine], src_force=force[mine], f0=20.0,
                                                   t0=3.0 * dt, rec_nodes=rec)
        assert rel_l2(uu[q], ref_u) <= 2e-5 and rel_l2(seis[q], ref_seis) <= 1e-4
