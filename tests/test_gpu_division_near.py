"""The one-launch attempt kernel on a node of high degree: more near partners than the tasks that share
them, in every part of the list (children, grandchildren, siblings). Tolerance: the 1e-12 that the
attempt's other sizes are held to against the oracle."""
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


@pytest.mark.parametrize("n", [13, 25, 45, 160])
@pytest.mark.parametrize("cluster", [1, 8])
@pytest.mark.parametrize("n_d", [1, 2])
def test_attempt_with_a_node_of_twelve_neighbours(n, cluster, n_d):
    m, r, v = W.plummer(n, 17)
    r = r + 20.0
    g = (1.0 + 5.0 ** 0.5) / 2.0
    ico = np.array([(0, a, b * g) for a in (-1, 1) for b in (-1, 1)], float)
    ico = np.concatenate([ico, ico[:, [1, 2, 0]], ico[:, [2, 0, 1]]]) * (1.0 + 1e-3 * np.arange(12))[:, None]
    r[0] = 0.0
    r[1:13] = ico
    r[13:25] = 1.4 * ico[:max(0, min(12, n - 13))]
    it = M.Integrator(m, r, v, division_schedule=3, division_cluster=cluster, n_d=n_d)
    o = O.System(m, r, v, n_d=n_d)
    gs, os_ = it.attempt(1e-3), o.attempt(1e-3)
    it.close()
    for key in ("r", "v"):
        assert np.abs(gs[key] - os_[key]).max() < 1e-12 * np.abs(os_[key]).max()
    assert abs(gs["t"] - os_["t"]) <= 1e-12 * abs(os_["t"])
