"""The surrogate's kernels where the networks of the other tests do not reach: the general tcgen05
kernels (sizes off the packed path's granules) over several tiles and channel chunks each way,
packed layers of odd lengths, and the wait limits of the packed kernels. Bars are those of
test_gpu_surrogate.py: outputs 2e-3 and loss 1e-3 against the FP64 oracle network that rounds the
same operands; gradients 1.5e-2 against the network without rounding, and 2e-3 against the mma.sync
kernels. (Against the rounding oracle a gradient of few samples can differ by more than 2e-3, for
both kinds of kernels alike, to 1e-5 of each other: a backward operand an ulp apart flips a bfloat16
rounding, 2^-8, and with two samples a few such flips do not average out.)"""
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
    a = np.asarray(a, np.float64)
    return float(np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300))


def oracle_net(spec, flat, rounding):
    from oracle import surrogate_oracle as so
    params = {}
    for name, arr in spec.split(flat.astype(np.float64)).items():
        params[name] = so.bf16_round(arr) if name[0] in "WC" else arr
    stages = list(zip((spec.c0,) + tuple(spec.stage_cout[:-1]), spec.stage_cout, spec.stage_up))
    return so.Surrogate(params, spec.c0, spec.l0, stages, spec.contract, bf16_operands=rounding)


def problem(spec, batch):
    flat = spec.init_params(5)
    flat += inputs.uniform(6, flat.shape, -0.05, 0.05).astype(np.float32)  # nonzero biases
    x = inputs.uniform(7, (batch, 9), -1, 1).astype(np.float32)
    t = inputs.uniform(8, (batch, spec.out_c, spec.out_l), -1, 1).astype(np.float32)
    return flat, x, t


# a last stage that is not contracted; one of 48 output channels; 640 hidden units, 100 seed channels
@pytest.mark.parametrize("hidden,c0,l0,cout,up,contract,batch", [
    (80, 40, 37, (100, 300), (2, 2), 0, 5),
    (64, 64, 130, (96, 6 * 48), (1, 1), 6, 3),
    (640, 100, 33, (136, 64), (2, 1), 2, 131),
])
def test_general_kernels_over_several_tiles(hidden, c0, l0, cout, up, contract, batch):
    check(hidden, c0, l0, cout, up, contract, batch)


# packed: lengths 13 and 26, 65, 127 and 254
@pytest.mark.parametrize("c0,l0,cout,up,contract,batch", [
    (64, 13, (32, 3 * 32), (2, 1), 3, 4),
    (64, 65, (64, 64), (1, 1), 2, 2),
    (64, 127, (32, 32, 32), (2, 1, 1), 1, 2),
])
def test_packed_layers_of_odd_lengths(c0, l0, cout, up, contract, batch):
    check(64, c0, l0, cout, up, contract, batch)


def check(hidden, c0, l0, cout, up, contract, batch):
    from paper_2606_12850_gb300 import surrogate
    spec = surrogate.Spec(in_dim=9, hidden=hidden, c0=c0, l0=l0, stage_cout=cout, stage_up=up, contract=contract)
    flat, x, t = problem(spec, batch)
    xd, td = torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda()
    m = surrogate.Model(spec, max_batch=batch)
    m.set_params(flat)
    got = []
    for product in (1, 0):
        m.product = product
        y = torch.full((batch, spec.out_c, spec.out_l), float("nan"), device="cuda")
        torch.cuda.synchronize()
        loss = m.loss_grad(xd, td)
        grads = spec.split(m.get_grads())
        m.forward(xd, y)
        m.sync()
        got.append((y.cpu().numpy(), loss, grads))
    (y, loss, grads), (y0, _, grads0) = got
    net = oracle_net(spec, flat, True)
    assert rel_l2(y, net.forward(x.astype(np.float64))[0]) <= 2e-3
    assert rel_l2(y, y0.astype(np.float64)) <= 2e-3
    ref_loss, _ = net.backward(x.astype(np.float64), t.astype(np.float64))
    assert abs(loss - ref_loss) <= 1e-3 * ref_loss
    _, exact = oracle_net(spec, flat, False).backward(x.astype(np.float64), t.astype(np.float64))
    for name in exact:
        assert rel_l2(grads[name], exact[name]) <= 1.5e-2, name
        assert rel_l2(grads[name], grads0[name].astype(np.float64)) <= 2e-3, name


@pytest.mark.parametrize("call", ["forward", "loss_grad"])
def test_packed_wait_limits_report_timeout(call):
    """Every packed kernel of a pass waits for an mbarrier phase nothing completes, gives up after
    its limit and leaves; the call (or the next sync) reports SEM_ETIMEOUT, and with the test
    switched off the same model computes what a fresh one does."""
    from paper_2606_12850_gb300 import surrogate
    spec = surrogate.Spec(in_dim=9, hidden=64, c0=16, l0=100, stage_cout=(32, 96, 2 * 64), stage_up=(2, 2, 1), contract=2)
    flat, x, t = problem(spec, 3)
    xd, td = torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda()

    def use(m):
        y = torch.zeros((3, spec.out_c, spec.out_l), device="cuda")
        torch.cuda.synchronize()
        if call == "forward":
            m.forward(xd, y)
            m.sync()
            return y.cpu().numpy()
        loss = m.loss_grad(xd, td)
        return np.append(m.get_grads(), loss)

    m = surrogate.Model(spec, max_batch=4)
    m.set_params(flat)
    m.set_option(surrogate.SG_OPT_STALL_TEST, 1)
    with pytest.raises(sem.SemError) as info:
        use(m)
    assert info.value.code == -5 and "timed out" in str(info.value)
    m.set_option(surrogate.SG_OPT_STALL_TEST, 0)
    fresh = surrogate.Model(spec, max_batch=4)
    fresh.set_params(flat)
    assert np.array_equal(use(m), use(fresh))
