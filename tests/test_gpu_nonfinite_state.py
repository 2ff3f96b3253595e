"""A state set to values that leave every distance undefined or infinite: the next step fails with
NO_CONVERGENCE, whatever builds the tree, and the context goes on from a good state."""
import numpy as np
import pytest

from paper_2001_03180_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA GPU", allow_module_level=True)

from paper_2001_03180_gb300 import build as B  # noqa: E402

B.build()
from paper_2001_03180_gb300 import mstar as M  # noqa: E402


@pytest.mark.parametrize("method,nsub", [(0, 0), (1, 0), (1, 1), (1, 300)])
@pytest.mark.parametrize("n", [40, 600, 3001])
def test_step_fails_and_the_context_recovers(n, method, nsub):
    m, r, v = W.plummer(n, 53)
    g = M.Integrator(m, r, v, mst_method=method, mst_nsub=min(nsub, n), max_halvings=3)
    H = 1e-6
    ref = g.attempt(H)
    for bodies, value in (([0], np.nan), ([n // 2, n - 1], np.nan), (list(range(n)), np.nan), ([3], np.inf),
                          ([3], -np.inf), (list(range(0, n, 2)), 1e200)):
        rb = r.copy()
        rb[bodies] = value
        g.set_state(0.0, rb, v)
        root, parent, level, _ = g.mst(with_order=False)
        # whatever the tree, it is one: each parent is a level nearer the root
        others = np.arange(n) != root
        assert parent[root] == -1 and level[root] == 0
        assert (parent[others] >= 0).all() and (parent < n).all()
        assert (level[others] == level[parent[others]] + 1).all()
        rc, _ = g.step(1.0, max_steps=1, check=False)
        assert rc == M.MSTAR_ERR_NO_CONVERGENCE
    g.set_state(0.0, r, v)
    a = g.attempt(H)
    g.close()
    assert np.allclose(a["r"], ref["r"], rtol=0, atol=1e-13) and np.allclose(a["v"], ref["v"], rtol=0, atol=1e-12)
