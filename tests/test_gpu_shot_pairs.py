"""Several shots at the edges of the rule that sweeps them in pairs (csrc/sem_capi.cpp, pair_rule:
up to NGLL 6, not at 3; even counts, odd ones from 13 on): under the default every shot equals its
own single-shot run to the batched bar, 2e-5 relative L2, and the default can be set again."""
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
    b = np.asarray(b, np.float64)
    return float(np.linalg.norm(np.asarray(a, np.float64) - b) / np.linalg.norm(b))


STEPS = 25


def setup(ngll, shots):
    w, pos = inputs.batched_layered_cube(n=3, ngll=ngll, nshots=shots, nsteps=STEPS)
    s = sem.setup_workload(w)
    nodes = sem.sem_locate_nodes(s.ctx, pos)
    sem.sem_set_shots(s.ctx, shots)
    sem.sem_set_shot_sources(s.ctx, np.arange(shots), nodes, np.tile([0.0, 5e9, 1e10], (shots, 1)), w.f0, 0.0)
    return w, s, nodes


def run(s):
    sem.sem_set_state(s.ctx)
    return sem.sem_run(s.ctx, STEPS), sem.sem_get_state(s.ctx, want=(True, False, False))[0]


@pytest.mark.parametrize("ngll,shots", [(2, 2), (2, 5), (3, 12), (3, 13), (5, 11), (5, 13), (5, 14), (6, 15), (7, 4), (7, 13)])
def test_default_rule_matches_single_shots(ngll, shots):
    w, s, nodes = setup(ngll, shots)
    seis, u = run(s)
    for q in sorted({0, 1, shots // 2, shots - 1}):
        p = sem.setup_workload(w, src_nodes=nodes[q:q + 1], rec_nodes=s.rec_nodes)
        sem.sem_set_source_nodes(p.ctx, nodes[q:q + 1], [[0.0, 5e9, 1e10]], w.f0, 0.0)
        one = run(p)
        assert rel_l2(seis[q], one[0]) <= 2e-5 and rel_l2(u[q], one[1]) <= 2e-5


@pytest.mark.parametrize("ngll,shots,pairs", [(5, 4, 1), (5, 5, 0), (5, 13, 1), (7, 4, 0)])
def test_default_rule_can_be_set_again(ngll, shots, pairs):
    """Value 2 after 0 and 1; the form the rule takes gives the default's results bit for bit."""
    _, s, _ = setup(ngll, shots)
    default = run(s)
    out = {}
    for value in (0, 1, 2):
        sem.sem_set_option(s.ctx, sem.SEM_OPT_SHOT_PAIRS, value)
        out[value] = run(s)
    for a, b, c in zip(default, out[2], out[pairs]):
        assert np.array_equal(a, b) and np.array_equal(a, c)
    for value in (-1, 3):
        with pytest.raises(sem.SemError):
            sem.sem_set_option(s.ctx, sem.SEM_OPT_SHOT_PAIRS, value)
