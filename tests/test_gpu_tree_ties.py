"""Trees of tied inputs: exact ties end the parallel rounds part-way through, wherever they are seen,
and the sequential builders take over; the tree is the oracle's."""
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

O.set_threads(16)


def half_lattice(n):
    """A Plummer sphere whose last third is a cubic lattice beside it: most subgraphs and many
    vertices have no tie, some have several, and the rounds meet them late."""
    m, r, v = W.plummer(n, 41)
    k = n // 3
    e = int(np.ceil(k ** (1.0 / 3.0)))
    g = np.stack(np.meshgrid(*[np.arange(float(e))] * 3, indexing="ij"), axis=-1).reshape(-1, 3)[:k]
    r[n - k:] = 0.5 * g + 8.0
    return m, r, v


def lattice(n):
    e = int(np.ceil(n ** (1.0 / 3.0)))
    g = np.stack(np.meshgrid(*[np.arange(float(e))] * 3, indexing="ij"), axis=-1).reshape(-1, 3)[:n]
    return np.ones(n), g, np.zeros((n, 3))


@pytest.mark.parametrize("make", [half_lattice, lattice])
@pytest.mark.parametrize("n,nsub", [(900, 0), (900, 300), (3001, 0), (3001, 1024), (8000, 1024)])
def test_divide_and_conquer_tree(make, n, nsub):
    m, r, v = make(n)
    g = M.Integrator(m, r, v, mst_method=1, mst_nsub=nsub)
    for _ in range(3):  # the same context again: its rounds are issued ahead of the first check
        root, par, lev, _ = g.mst(with_order=False)
        ro, po, lo, _, _, _ = O.dc_mst(g.state()["r"], nsub)
        assert root == ro and np.array_equal(par, po) and np.array_equal(lev, lo)
        g.set_state(0.0, r, v)
    g.close()


@pytest.mark.parametrize("make", [half_lattice, lattice])
@pytest.mark.parametrize("n", [512, 900, 3001, 8000])
def test_step_tree_after_another_system(make, n):
    """The step's tree of a tied system in a context whose scratch holds another system's sums."""
    m, r, v = make(n)
    _, r0, v0 = W.plummer(n, 43)
    g = M.Integrator(m, r0, v0)
    for _ in range(2):
        g.set_state(0.0, r0, v0)
        g.attempt(1e-6)
        g.set_state(0.0, r, v)
        root, par, lev, _ = g.mst(with_order=False)
        ro, po, lo, _ = O.prim(g.state()["r"])
        assert root == ro and np.array_equal(par, po) and np.array_equal(lev, lo)
    g.close()
