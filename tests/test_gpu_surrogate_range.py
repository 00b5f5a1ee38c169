"""The packed training step over the whole range the surrogate takes: output widths past the
general loss kernel's block count, and errors whose squares leave float32's range. Against the
FP64 oracle network that rounds the same operands. Bars: relative L2 2e-3 for gradients, 1e-3 for
the loss (those of the other surrogate tests: bfloat16 rounding boundaries)."""
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


def test_outputs_wider_than_the_general_loss_kernel_s_blocks():
    """610 column blocks of the last convolution, each with a loss value of its own."""
    from paper_2606_12850_gb300 import surrogate
    spec = surrogate.Spec(in_dim=9, hidden=64, c0=16, l0=4, stage_cout=(32 * 610,), stage_up=(1,), contract=1)
    m = surrogate.Model(spec, max_batch=2)
    flat = spec.init_params(5)
    m.set_params(flat)
    x = inputs.uniform(7, (2, 9), -1, 1).astype(np.float32)
    t = inputs.uniform(8, (2, spec.out_c, spec.out_l), -1, 1).astype(np.float32)
    loss = m.loss_grad(torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda())
    grads = spec.split(m.get_grads())
    ref_loss, ref_g = oracle_net(spec, flat).backward(x.astype(np.float64), t.astype(np.float64))
    assert abs(loss - ref_loss) <= 1e-3 * ref_loss
    for name in ref_g:
        assert rel_l2(grads[name], ref_g[name]) <= 2e-3, name


@pytest.mark.parametrize("scale", [1e21, 1e-22])
def test_loss_of_errors_whose_squares_leave_float32(scale):
    """Targets and last layer of this scale: the squared errors, 1e42 or 1e-44, are outside
    float32's normal range, their mean is an ordinary float64 number (the gradients of the layers
    below the last are outside float32 at the small scale in any case)."""
    from paper_2606_12850_gb300 import surrogate
    spec = surrogate.Spec(in_dim=9, hidden=64, c0=16, l0=20, stage_cout=(32, 3 * 32), stage_up=(2, 1), contract=3)
    m = surrogate.Model(spec, max_batch=3)
    flat = spec.init_params(5)
    last = spec.split(flat)["C1"].size + spec.split(flat)["c1"].size
    flat[-last:] = inputs.uniform(6, (last,), -0.1, 0.1) * min(scale, 1.0)
    m.set_params(flat)
    x = inputs.uniform(7, (3, 9), -1, 1).astype(np.float32)
    t = (inputs.uniform(8, (3, spec.out_c, spec.out_l), -1, 1) * scale).astype(np.float32)
    loss = m.loss_grad(torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda())
    grads = spec.split(m.get_grads())
    ref_loss, ref_g = oracle_net(spec, flat).backward(x.astype(np.float64), t.astype(np.float64))
    assert ref_loss > 0 and abs(loss - ref_loss) <= 1e-3 * ref_loss
    for name in ("C1", "c1"):
        assert rel_l2(grads[name], ref_g[name]) <= 2e-3, name
