"""Backpropagation through seismograms of a simulation whose ``gradient(G)`` is redefined (weights
of the residual, a preconditioner): the redefined one is called, with G alone, and its host arrays
are the gradients."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2606_12850_gb300 import adjoint, build, inputs, sem  # noqa: E402

pytestmark = pytest.mark.gpu


class Halved(adjoint.Simulation):
    def gradient(self, G):
        return tuple(0.5 * g for g in super().gradient(G))


@pytest.mark.parametrize("redefined", ["subclass", "object"])
def test_redefined_gradient_is_used(redefined):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    w = inputs.layered_cube(4, n=2, side=600.0, nrec_side=2)
    s = sem.setup_workload(w)
    mu = np.asarray(w.rho * w.vs * w.vs, np.float32)
    mats = [np.asarray(w.rho, np.float32), np.asarray(w.rho * w.vp * w.vp, np.float32) - np.float32(4 / 3) * mu, mu]
    grads = []
    for cls in (adjoint.Simulation, Halved if redefined == "subclass" else adjoint.Simulation):
        sim = cls(s.ctx, s.dt, 40, keep_all=True)
        if grads and redefined == "object":
            plain = sim.gradient
            sim.gradient = lambda G: tuple(0.5 * g for g in plain(G))
        leaf = [torch.from_numpy(a).cuda().requires_grad_(True) for a in mats]
        seis = adjoint.Seismograms.apply(*leaf, sim)
        (1e12 * seis).sum().backward()
        grads.append([x.grad.cpu().numpy() for x in leaf])
    for g, h in zip(*grads):
        assert np.any(g != 0.0)
        np.testing.assert_array_equal(h, 0.5 * g)  # halving is exact, also after rounding to float32
