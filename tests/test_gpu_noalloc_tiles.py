"""mstar_accelerations_noalloc at the edges of its tile sizes and arithmetics, against long double sums.

Tolerance: a component is the sum of n terms, each within 8 u (u = 2^-53) of m_j d / r^3, added in
binary64 (or finer, in integers) in chains of at most 32 steps, 8 warps and 16 slots: the sum errs
by at most (8 + 32 + 8 + 16 + 2) u sum |f_ij| = 66 u sum |f_ij| with the product by G; 80 u is taken.
U adds chains of 32, 5, 16, 2 and 10 terms: the same bound serves.
"""
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


def run(m, r, G):
    dev = torch.device("cuda")
    mt = torch.tensor(m, dtype=torch.float64, device=dev)
    rt = torch.tensor(r, dtype=torch.float64, device=dev)
    a = torch.full_like(rt, 7.0)
    U = torch.empty(1, dtype=torch.float64, device=dev)
    assert M.mstar_accelerations_noalloc(len(m), mt, rt, G, a, U, torch.cuda.current_stream().cuda_stream) == M.MSTAR_OK
    torch.cuda.synchronize()
    return a.cpu().numpy(), float(U.item())


@pytest.mark.parametrize("kind", ["plain", "spectrum", "signs", "close", "flat"])
@pytest.mark.parametrize("n", [2, 3, 31, 32, 33, 64, 65, 511, 512, 513, 1024, 1025, 1151, 2048])
def test_sums_at_tile_edges(n, kind):
    s = W.Stream(23, n)
    r = np.stack([s.uniform(n) - 0.5 for _ in range(3)], 1)
    m = np.full(n, 1.0 / n)
    if kind == "spectrum":
        m = m * 10.0 ** (-3.0 * s.uniform(n))
    elif kind == "signs":      # massless and negative sources: FP64 throughout
        m[::3] = 0.0
        m[1::5] *= -1.0
    elif kind == "close":      # pairs far closer than the integer window
        r[n // 2:] = r[:n - n // 2] + 1e-6 * (1.0 + s.uniform(n - n // 2))[:, None]
    elif kind == "flat":
        r[:, 1] *= 1e-7
    G = 1.75
    a, U = run(m, r, G)
    rl, ml = r.astype(np.longdouble), m.astype(np.longdouble)
    rows = np.unique(np.linspace(0, n - 1, min(n, 64)).astype(int))
    d = rl[None] - rl[rows, None]
    r2 = (d * d).sum(-1)
    r2[np.arange(len(rows)), rows] = 1.0
    f = ml[None, :, None] * d / (r2 * np.sqrt(r2))[..., None]
    # a direction's terms are bounded with the whole force: integers share one unit in all three
    bound = np.abs(ml[None] / r2).sum(1) - np.abs(ml[rows])
    assert (np.abs(a[rows] - G * f.sum(1)).max(1) <= 80 * 2.0 ** -53 * G * bound).all()
    d = r[None] - r[:, None]
    dist = np.sqrt((d * d).sum(-1))
    np.fill_diagonal(dist, np.inf)
    w = m[:, None] * m[None] / dist
    # the float64 reference itself: pairwise sums, below 32 u
    assert abs(U - G * 0.5 * w.sum()) <= (80 + 32) * 2.0 ** -53 * G * 0.5 * np.abs(w).sum()


@pytest.mark.parametrize("n", [40, 600, 1100])
def test_coincident_and_non_finite_bodies_give_nan(n):
    s = W.Stream(29, n)
    r = np.stack([s.uniform(n) for _ in range(3)], 1)
    m = np.full(n, 1.0)
    rc = r.copy()
    rc[n - 1] = rc[3]
    a, U = run(m, rc, 1.0)
    assert np.isnan(a[[3, n - 1]]).all() and not U < 1e150  # 1/r of a zero distance: about 2^512, as ever
    assert np.isfinite(np.delete(a, [3, n - 1], axis=0)).all()
    rn = r.copy()
    rn[5, 1] = np.nan
    a, U = run(m, rn, 1.0)
    assert np.isnan(U) and np.isnan(a[:, 1]).all()
