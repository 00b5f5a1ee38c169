"""The surrogate's packed tensor-core path (sizes of 64-feature and 32-channel granules) against
the FP64 oracle network that rounds the same operands, at the edges of its tiles: time axes
shorter than, just above and several times the 128-row tile, with and without upsampling,
batches of one and just above 128, and several contraction counts. Bars: relative L2 2e-3 for
outputs and gradients, 1e-3 for the loss (an operand whose float32 and float64 values straddle a
bfloat16 rounding boundary rounds differently on the two sides). The general kernels
(SG_OPT_PRODUCT 0) must agree with it to the same bar."""
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


def oracle_net(spec, flat):
    from oracle import surrogate_oracle as so
    params = {}
    for name, arr in spec.split(flat.astype(np.float64)).items():
        params[name] = so.bf16_round(arr) if name[0] in "WC" else arr
    stages = list(zip((spec.c0,) + tuple(spec.stage_cout[:-1]), spec.stage_cout, spec.stage_up))
    return so.Surrogate(params, spec.c0, spec.l0, stages, spec.contract, bf16_operands=True)


@pytest.mark.parametrize("c0,l0,cout,up,contract,batch", [
    (16, 20, (32, 64, 6 * 32), (2, 1, 1), 6, 129),
    (32, 130, (32, 2 * 32), (1, 1), 2, 3),
    (16, 100, (32, 96, 6 * 64), (2, 2, 1), 6, 1),
    (48, 64, (96, 5 * 96), (2, 1), 5, 5),
])
def test_packed_network_matches_oracle(c0, l0, cout, up, contract, batch):
    from paper_2606_12850_gb300 import surrogate
    spec = surrogate.Spec(in_dim=9, hidden=64, c0=c0, l0=l0, stage_cout=cout, stage_up=up, contract=contract)
    m = surrogate.Model(spec, max_batch=max(2, batch))
    flat = spec.init_params(5)
    flat += inputs.uniform(6, flat.shape, -0.05, 0.05).astype(np.float32)  # nonzero biases
    m.set_params(flat)
    x = inputs.uniform(7, (batch, 9), -1, 1).astype(np.float32)
    t = inputs.uniform(8, (batch, spec.out_c, spec.out_l), -1, 1).astype(np.float32)
    xd, td = torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda()
    y = torch.full((batch, spec.out_c, spec.out_l), float("nan"), device="cuda")
    torch.cuda.synchronize()
    net = oracle_net(spec, flat)
    ref, _ = net.forward(x.astype(np.float64))
    loss = m.loss_grad(xd, td)
    grads = spec.split(m.get_grads())
    m.forward(xd, y)
    m.sync()
    assert rel_l2(y.cpu().numpy(), ref) <= 2e-3
    ref_loss, ref_g = net.backward(x.astype(np.float64), t.astype(np.float64))
    assert abs(loss - ref_loss) <= 1e-3 * ref_loss
    for name in ref_g:
        assert rel_l2(grads[name], ref_g[name]) <= 2e-3, name
    m.product = 0
    z = torch.empty_like(y)
    m.forward(xd, z)
    m.sync()
    assert rel_l2(z.cpu().numpy(), y.cpu().numpy().astype(np.float64)) <= 2e-3
