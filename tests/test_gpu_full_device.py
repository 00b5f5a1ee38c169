"""Calls that need no device memory of their own, or can do without the part they lack, on a device
that other arrays fill up."""
import contextlib
import gc

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
    """Within it, other arrays hold the free device memory but for ``leave`` bytes and less than 12 MB
    more (smaller arrays would come from segments of 20 MB)."""
    gc.collect()  # contexts of earlier tests, held by tracebacks, must not give memory back within it
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    held = []
    part = 1
    while (free := (torch.cuda.mem_get_info()[0] - leave) // part // (2 << 20) * (2 << 20)) >= 12 << 20:
        try:
            held.append(torch.empty(free, dtype=torch.uint8, device="cuda"))
        except torch.OutOfMemoryError:
            part *= 2
    try:
        yield
    finally:
        held.clear()
        torch.cuda.empty_cache()


def test_gradients_to_the_host():
    w = inputs.layered_cube(5, n=24, side=2000.0, nrec_side=2)  # 14 MB of float64 a gradient
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
    the model is created and the general tcgen05 kernels take its calls. Their outputs are the packed
    kernels' bit for bit (the same operands, K order and roundings); gradients differ in the order of
    float32 sums."""
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
    assert np.array_equal(ref[2], got[2])
    for name, a in spec.split(ref[3]).items():
        b = spec.split(got[3])[name]
        assert np.linalg.norm(a - b) <= 2e-3 * np.linalg.norm(a), name


def rel_l2(a, b):
    return float(np.linalg.norm(a.astype(np.float64) - b) / np.linalg.norm(b))


def test_shots_without_room_for_the_sweep_s_partials():
    """32 shots whose fields fit (422 MB) and whose partial sums (91 MB) do not."""
    w = inputs.layered_cube(5, n=16, side=2000.0, nrec_side=2)
    shots, out = 32, []
    pos = inputs.uniform(3, (shots, 3), 500.0, 1500.0)
    for tight in (False, True):
        s = sem.setup_workload(w)
        nodes = sem.sem_locate_nodes(s.ctx, pos)
        sem.sem_run(s.ctx, 2)  # loads the kernels of the shots' set-up
        if tight:
            with full_device(leave=48 * (shots - 1) * w.mesh.nglob + (32 << 20)):
                sem.sem_set_shots(s.ctx, shots)
        else:
            sem.sem_set_shots(s.ctx, shots)
        sem.sem_set_shot_sources(s.ctx, np.arange(shots), nodes, np.tile([0.0, 1e10, 1e10], (shots, 1)), w.f0, 0.0)
        sem.sem_set_state(s.ctx)
        seis = sem.sem_run(s.ctx, 13)
        u = sem.sem_get_state(s.ctx, want=(True, False, False))[0]
        out.append((sem.sem_info(s.ctx)["device_bytes"], seis, u))
    assert out[0][0] - out[1][0] > 80 << 20
    assert rel_l2(out[1][1], out[0][1]) <= 2e-5 and rel_l2(out[1][2], out[0][2]) <= 2e-5


def test_mesh_without_room_for_the_sweep_s_partials():
    """A mesh of which only the partial sums (25 MB) do not fit: steps by the persistent sweep, which
    adds in the same order, f = -K u on caller arrays by the element kernel, the adjoint."""
    w = inputs.layered_cube(5, n=32, side=4000.0, nrec_side=2)
    sem.setup_workload(inputs.layered_cube(5, n=2, side=400.0, nrec_side=2))  # loads the kernels
    out, need = [], None
    for tight in (False, True):
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        before = torch.cuda.mem_get_info()[0]
        ctx = sem.sem_create(5, 0)
        if tight:
            with full_device(leave=need - (18 << 20)):
                sem.sem_set_mesh_corners(ctx, w.mesh.ibool, w.mesh.ctrl, w.mesh.nglob)
        else:
            sem.sem_set_mesh_corners(ctx, w.mesh.ibool, w.mesh.ctrl, w.mesh.nglob)
            need = before - torch.cuda.mem_get_info()[0]
        held = sem.sem_info(ctx)["device_bytes"]
        sem.sem_set_material(ctx, w.rho, w.vp, w.vs)
        sem.sem_set_dt(ctx, sem.sem_suggest_dt(ctx, 0.3))
        node = sem.sem_locate_nodes(ctx, w.source_xyz)
        sem.sem_set_source_nodes(ctx, node, w.source_force, w.f0, 0.0)
        sem.sem_set_receiver_nodes(ctx, node)
        sem.sem_set_state(ctx)
        seis = sem.sem_run(ctx, 13)
        u = sem.sem_get_state(ctx, want=(True, False, False))[0]
        field = torch.from_numpy(inputs.random_field(w.mesh.nglob, 6)).cuda()
        f = torch.empty_like(field)
        snaps = field[None].repeat(4, 1, 1) * torch.arange(4, device="cuda")[:, None, None]
        G = torch.ones((2, len(node), 3), device="cuda")
        torch.cuda.synchronize()
        sem.sem_apply_stiffness(ctx, field, f)
        sem.sem_sync(ctx)
        sem.sem_adjoint_begin(ctx)
        sem.sem_adjoint_segment(ctx, 2, G, snaps)
        out.append((held, seis, u, f.cpu().numpy(), sem.sem_adjoint_gradients(ctx)))
        del ctx, field, f, snaps
    a, b = out
    assert a[0] - b[0] > 20 << 20
    assert np.array_equal(a[1], b[1]) and np.array_equal(a[2], b[2]) and np.any(a[1] != 0)
    assert rel_l2(b[3], a[3]) <= 1e-6
    for x, y in zip(a[4], b[4]):
        assert rel_l2(y, x) <= 1e-5


@pytest.mark.parametrize("what", ["receivers", "sources", "shots", "mesh"])
def test_set_up_call_that_runs_out_of_memory_leaves_a_usable_context(what):
    """Receivers, sources, shots or a mesh that do not fit: the call reports it, and the context
    steps without what it could not take (one shot again; no receivers or sources; no mesh)."""
    w = inputs.layered_cube(5, n=32, side=2000.0, nrec_side=2)
    nglob, every = w.mesh.nglob, np.arange(w.mesh.nglob, dtype=np.int32)
    u = inputs.random_field(nglob, 6, scale=1e-3)
    big = inputs.layered_cube(5, n=48, side=2000.0, nrec_side=2).mesh if what == "mesh" else None
    s = sem.setup_workload(w)

    def steps():
        sem.sem_set_state(s.ctx, u)
        return sem.sem_run(s.ctx, 13), sem.sem_get_state(s.ctx, want=(True, False, False))[0]

    def again():
        sem.sem_set_source_nodes(s.ctx, s.src_nodes, w.source_force, w.f0, w.t0)
        sem.sem_set_receiver_nodes(s.ctx, s.rec_nodes)

    both = steps()
    sem.sem_set_source_nodes(s.ctx, [], np.zeros((0, 3)), w.f0, 0.0)
    sourceless = steps()
    again()
    steps()  # graphs that hold the present lists
    with full_device():
        with pytest.raises(sem.SemError) as info:
            if what == "receivers":
                sem.sem_set_receiver_nodes(s.ctx, np.tile(every, 8))
            elif what == "sources":
                sem.sem_set_source_nodes(s.ctx, every, np.ones((nglob, 3)), w.f0, 0.0)
            elif what == "shots":
                sem.sem_set_shots(s.ctx, 8)
            else:
                sem.sem_set_mesh_corners(s.ctx, big.ibool, big.ctrl, big.nglob)
    assert info.value.code == -2
    if what == "mesh":
        with pytest.raises(sem.SemError) as info:
            sem.sem_step(s.ctx, 1)
        assert info.value.code == -4
        return
    assert s.ctx.shots == 1
    seis, end = steps()
    if what == "receivers":
        assert seis is None and np.array_equal(end, both[1])
    else:  # none of the old sources either
        assert np.array_equal(seis, sourceless[0]) and np.array_equal(end, sourceless[1])
    assert not np.array_equal(both[1], sourceless[1])
    again()  # and the context takes them again
    for a, b in zip(steps(), both):
        assert np.array_equal(a, b)
