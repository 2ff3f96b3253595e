"""Prim's tree of small systems (one warp up to 96 bodies, one vertex per thread up to 512): root,
parents, levels and order equal the oracle's, index by index, with generic positions, with every
distance tied, and with distances closer than the float intervals resolve."""
import numpy as np
import pytest

import oracle as O
from paper_2001_03180_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA GPU", allow_module_level=True)

from paper_2001_03180_gb300 import build as B  # noqa: E402

B.build()
from paper_2001_03180_gb300 import mstar as M  # noqa: E402


@pytest.mark.parametrize("kind", ["generic", "lattice", "near_ties", "hierarchy"])
@pytest.mark.parametrize("n", [2, 3, 31, 32, 33, 64, 65, 96, 97, 128, 129, 160, 257, 511, 512])
def test_tree_matches_the_oracle(n, kind):
    s = W.Stream(31, n)
    r = np.stack([s.uniform(n) - 0.5 for _ in range(3)], 1)
    if kind == "lattice":
        side = int(np.ceil(n ** (1 / 3)))
        r = np.array([(i % side, i // side % side, i // side // side) for i in range(n)], float)
    elif kind == "near_ties":   # a line of spacings equal to 1e-9
        r = np.zeros((n, 3))
        r[:, 0] = np.arange(n) + 1e-9 * s.uniform(n)
    elif kind == "hierarchy":   # separations from 1e-12 to 1 about distant centres
        r = r * 10.0 ** (-12.0 * s.uniform(n))[:, None] + np.round(4 * r)
    v = np.zeros_like(r)
    v[:, 1] = 1e-3 * s.uniform(n)
    g = M.Integrator(np.full(n, 1.0 / n), r, v)
    root, par, lev, order = g.mst()
    rs = g.state()["r"]
    g.close()
    want = O.prim(rs)
    assert root == want[0]
    assert np.array_equal(par, want[1]) and np.array_equal(lev, want[2]) and np.array_equal(order, want[3])
