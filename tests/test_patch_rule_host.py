"""The brick an order's mesh gets by default (csrc/sem_kernels.cu, patch_shape): at NGLL 5 the
cube of eight from 4000 elements on, the order's own brick below and at every other order."""
import numpy as np
import pytest

from paper_2606_12850_gb300 import build, inputs, sem


@pytest.fixture(scope="module", autouse=True)
def library():
    build.build()
    return sem.lib()


@pytest.mark.parametrize("ngll,dims,brick", [
    (5, (31, 43, 3), (1, 4, 2)),   # 3999
    (5, (25, 10, 16), (2, 2, 2)),  # 4000, a mesh the brick divides
    (5, (17, 17, 15), (2, 2, 2)),  # 4335, none of its sides
    (5, (4001, 1, 1), (2, 2, 2)),  # a row: bricks of two elements
    (4, (16, 16, 16), (4, 2, 2)),
    (7, (16, 16, 16), (1, 2, 2)),
])
def test_default_brick(ngll, dims, brick):
    m = inputs.structured_hex_mesh(dims, ngll, 1.0)
    patch, color, info = sem.sem_patch_plan(ngll, m.ibool, m.nglob)
    assert (info["bx"], info["by"], info["bz"]) == brick
    counts = np.bincount(patch, minlength=info["patches"])
    per = [min(b, d) for b, d in zip(brick, dims)]
    assert counts.min() >= 1 and counts.max() == int(np.prod(per))
    assert info["patches"] == int(np.prod([-(-d // b) for d, b in zip(dims, brick)]))
    # no two patches of a colour share a node
    nodes = np.asarray(m.ibool).reshape(patch.size, -1)
    pair = np.unique(np.stack([np.repeat(patch, nodes.shape[1]), nodes.ravel()], 1), axis=0)
    key = color[pair[:, 0]].astype(np.int64) * m.nglob + pair[:, 1]
    assert np.unique(key).size == key.size
