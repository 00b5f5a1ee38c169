"""Two surrogates of different sizes used from two threads at once: every call succeeds and gives
what the model gives alone, bit for bit (each has its own stream and buffers; the kernels'
shared-memory limit belongs to the process)."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2606_12850_gb300 import build, inputs  # noqa: E402

pytestmark = pytest.mark.gpu


def test_models_of_two_sizes_in_two_threads():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    from paper_2606_12850_gb300 import surrogate
    specs = [surrogate.Spec(in_dim=9, hidden=64, c0=16, l0=20, stage_cout=(32, 32), stage_up=(2, 1), contract=1),
             surrogate.Spec(in_dim=9, hidden=256, c0=64, l0=20, stage_cout=(96, 6 * 64), stage_up=(2, 1), contract=6)]
    work = []
    for k, spec in enumerate(specs):
        m = surrogate.Model(spec, max_batch=2)
        m.set_params(spec.init_params(5 + k))
        x = torch.from_numpy(inputs.uniform(7, (2, 9), -1, 1).astype(np.float32)).cuda()
        t = torch.from_numpy(inputs.uniform(8, (2, spec.out_c, spec.out_l), -1, 1).astype(np.float32)).cuda()
        y = torch.empty((2, spec.out_c, spec.out_l), device="cuda")
        torch.cuda.synchronize()
        m.forward(x, y)
        loss = m.loss_grad(x, t)  # waits for the model's stream
        work.append((m, x, t, y, y.cpu().numpy(), loss, m.get_grads()))
    errors = []

    def use(m, x, t, y, ref, loss, grads):
        try:
            for _ in range(10000):  # launches without waits between them
                m.forward(x, y)
            for _ in range(200):
                if m.loss_grad(x, t) != loss:
                    errors.append("loss")
            if not np.array_equal(y.cpu().numpy(), ref) or not np.array_equal(m.get_grads(), grads):
                errors.append("values")
        except Exception as e:  # noqa: BLE001  (reported below, in the main thread)
            errors.append(repr(e))

    threads = [threading.Thread(target=use, args=w) for w in work]
    for th in threads:
        th.start()
    for th in threads:
        th.join()
    assert not errors, errors[:3]
