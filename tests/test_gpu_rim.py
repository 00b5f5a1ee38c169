"""The one-launch patch sweep and its rim pass against the FP64 oracle, where they can go wrong:
sources and receivers on inner nodes, faces, edges and corners of the patches, meshes the
bricks do not divide, nodes where more than four patches meet (single-element patches), one
and several shots. Bars: the solver's wavefield 2e-5 and seismogram 1e-4 relative L2."""
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


def rel_l2(a, b):
    return float(np.linalg.norm(np.asarray(a, np.float64) - b) / np.linalg.norm(b))


@pytest.mark.parametrize("ngll,shape,shots,assembly", [(2, 0, 1, 0), (3, 0, 1, 0), (4, 0, 3, 0), (5, 0, 1, 0), (5, 1, 1, 0),
                                                       (5, 1, 3, 0), (5, 0, 2, 2), (8, 0, 1, 0), (10, 0, 1, 0)])
def test_sweep_and_rim_match_oracle(oracle, ngll, shape, shots, assembly):
    w = inputs.layered_cube(ngll, n=3, side=600.0, nrec_side=2)
    m = oracle.build_model(w)
    dt = m.cfl_dt(0.4)
    ctx = sem.sem_create(ngll, 0)
    if shape:  # patches of one element: eight of them meet at an interior vertex
        sem.sem_set_option(ctx, sem.SEM_OPT_PATCH_SHAPE, sem.patch_shape_code(1, 1, 1))
    sem.sem_set_option(ctx, sem.SEM_OPT_ASSEMBLY, assembly)
    sem.sem_set_mesh_corners(ctx, w.mesh.ibool, w.mesh.ctrl, w.mesh.nglob)
    sem.sem_set_material(ctx, w.rho, w.vp, w.vs)
    sem.sem_set_dt(ctx, dt)
    # element corners (rim nodes of every kind) and random nodes
    G = 3 * (ngll - 1) + 1
    lattice = np.arange(0, G, ngll - 1)
    corners = (lattice[:, None, None] * G * G + lattice[None, :, None] * G + lattice[None, None, :]).ravel()
    pick = np.unique(np.concatenate([corners, (inputs.uniform(3, (40,)) * w.mesh.nglob).astype(np.int64)]))
    src = pick[::5].astype(np.int32)
    force = inputs.uniform(4, (len(src), 3), -1e10, 1e10)
    rec = pick.astype(np.int32)
    t0 = 3.0 * dt
    sem.sem_set_shots(ctx, shots)
    sem.sem_set_shot_sources(ctx, np.arange(len(src)) % shots, src, force, 30.0, t0)
    sem.sem_set_receiver_nodes(ctx, rec)
    sem.sem_set_state(ctx)
    seis = sem.sem_run(ctx, 13).reshape(shots, len(rec), 3, 13)
    u = sem.sem_get_state(ctx, want=(True, False, False))[0].reshape(shots, -1, 3)
    for q in range(shots):
        mine = np.arange(len(src)) % shots == q
        ref_seis, ref_u, _, _ = oracle.newmark_run(m, dt, 13, src_nodes=src[mine], src_force=force[mine], f0=30.0, t0=t0,
                                                   rec_nodes=rec)
        assert rel_l2(u[q], ref_u) <= 2e-5
        assert rel_l2(seis[q], ref_seis) <= 1e-4


@pytest.mark.parametrize("ngll,shape", [(2, 0), (5, 0), (5, 1), (9, 0)])
def test_stiffness_on_caller_arrays_matches_internal(ngll, shape):
    """f = -K u on caller arrays equals the sweep on the solver's own layout bit for bit."""
    w = inputs.layered_cube(ngll, n=3, side=600.0, nrec_side=2)
    ctx = sem.sem_create(ngll, 0)
    if shape:
        sem.sem_set_option(ctx, sem.SEM_OPT_PATCH_SHAPE, sem.patch_shape_code(1, 1, 1))
    sem.sem_set_mesh_corners(ctx, w.mesh.ibool, w.mesh.ctrl, w.mesh.nglob)
    sem.sem_set_material(ctx, w.rho, w.vp, w.vs)
    perm = torch.from_numpy(sem.sem_node_order(ctx).astype(np.int64)).cuda()
    u = torch.from_numpy(inputs.random_field(w.mesh.nglob, 6)).cuda()
    f = torch.full_like(u, float("nan"))
    u4 = torch.zeros((w.mesh.nglob, 4), device="cuda")
    u4[:, :3] = u[perm]
    f4 = torch.full_like(u4, float("nan"))
    torch.cuda.synchronize()
    sem.sem_apply_stiffness(ctx, u, f)
    sem.sem_apply_stiffness_strided(ctx, u4, f4, 4)
    sem.sem_sync(ctx)
    assert torch.equal(f[perm], f4[:, :3])
