"""Batched systems whose pair blocks integers do not serve (thin discs, bodies far out, masses outside
the range): the attempt after the start evaluation sweeps them. One attempt against the oracle's, to
1e-12 as for the other batched systems, beside systems that stay in integers."""
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


def system(kind, n):
    m, r, v = W.plummer(n, 47)
    m, r, v = m.copy(), r.copy(), v.copy()
    if kind == "disc":
        r[:, 2] *= 1e-3
    elif kind == "far":
        r[::3] *= 2e3
    elif kind == "massive":
        m *= 2.0 ** 50
        v *= 2.0 ** 25
    return m, r, v


@pytest.mark.parametrize("schedule", [None, [1] * 7, [2] * 7, [4] * 7, [-1] * 7, [-2] * 7, [-4] * 7])
def test_attempts_match_the_oracle(schedule):
    systems, H = [], []
    for kind in ("disc", "plain", "far", "massive"):
        for n in (17, 31, 32, 33, 64, 97):
            m, r, v = system(kind, n)
            systems.append((m, r, v))
            # a time step of 2e-4 of the dynamical time of a sphere of this mass
            H.append(2e-4 / np.sqrt(m.sum()) * O.potential(m, O.com_shift(m, r)))
    b = M.Batch(systems, eta_gbs=1.0)
    if schedule is not None:
        b.set_schedule(schedule)
    b.set_H(np.array(H))
    st = b.step(1e9, launches=1)
    assert st["accepted"] == len(systems)
    S = b.state()
    b.close()
    rel = lambda x, y: float(np.abs(x - y).max() / np.abs(y).max())  # noqa: E731
    for s, (m, r, v) in enumerate(systems):
        a = O.System(m, r, v).attempt(H[s])
        assert rel(S["r"][s], a["r"]) < 1e-12 and rel(S["v"][s], a["v"]) < 1e-12, s
        assert abs(S["t"][s] - a["t"]) <= 1e-12 * abs(a["t"]), s
