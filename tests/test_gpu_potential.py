"""The force function of systems with one dominant mass, through every pair loop that sums it in
integers, against long double sums.

Tolerance of U (u = 2^-53): a term m_i m_j / r errs by at most 8 u of itself, a near pair's by 8 u
more (its separation is the sum of two rounded edge vectors, none longer than the separation). The 32
terms that a warp adds in integers err by at most 2 u of their sum together. The binary64 additions
after that form chains of at most 3 (warps), 9 (partial slots, four at a time, for n <= 800), 8 (near
partners), 2, 10 (a block) and 6 (the blocks) roundings, 38 in all: 56 u, and 64 u is taken. The
sums hold no cancellation, so the bound is relative, for any ratio of the masses. The same bound
holds for an acceleration, relative to the sum of its terms' magnitudes.

The batch gives U through the time of one short step from rest: with k_fix = 2 the physical time is
4/3 t_2 - 1/3 t_1, each t_k a sum of h / (T + B), B = U. That is 5/3 of U's relative error, of the
64 u above, and some roundings of the step itself, below 20 u: 128 u is taken.
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

U53 = 2.0 ** -53
LD = np.longdouble


def places(n):
    return [0, n // 2, n - 1]


def system(n, ratio, place):
    m, r, _ = W.plummer(n, 31)
    m = m.copy()
    m[place] *= ratio
    return m, r


def forces(m, r):
    """Accelerations, the sums of their terms' magnitudes and U, in long double."""
    m, r = m.astype(LD), r.astype(LD)
    d = r[None] - r[:, None]
    r2 = (d * d).sum(-1)
    np.fill_diagonal(r2, LD(1))
    dist = np.sqrt(r2)
    w = m[None] / (r2 * dist)
    np.fill_diagonal(w, LD(0))
    p = m[:, None] * m[None] / dist
    np.fill_diagonal(p, LD(0))
    return (w[..., None] * d).sum(1), (w * dist).sum(1), p.sum() / 2


def check(a, U, m, r):
    ae, bound, Ue = forces(m, r)
    assert abs(U - Ue) <= 64 * U53 * Ue, float(abs(U - Ue) / Ue / U53)
    if a is not None:
        assert (np.abs(a - ae).max(1) <= 64 * U53 * bound).all()


@pytest.mark.parametrize("ratio", [1e4, 1e8, 1e12, 1e18])
@pytest.mark.parametrize("n,tile", [(32, 0), (33, 0), (160, 0), (161, 0), (512, 0), (513, 0), (768, 0), (769, 0),
                                    (641, 64), (641, 128)])
def test_context_sums(n, tile, ratio):
    for place in places(n):
        m, r = system(n, ratio, place)
        for n_d in (0, 2):
            g = M.Integrator(m, r, np.zeros_like(r), pair_tile=tile, n_d=n_d)
            a, U = g.accelerations()
            e = g.energy()
            rs = g.state()["r"]
            g.close()
            check(a, U, m, rs)
            check(None, e["U"], m, rs)


@pytest.mark.parametrize("ratio", [1e4, 1e8, 1e12, 1e18])
@pytest.mark.parametrize("n", [32, 33, 512, 513, 1024, 1025])
def test_allocation_free_sums(n, ratio):
    dev = torch.device("cuda")
    for place in places(n):
        m, r = system(n, ratio, place)
        a = torch.empty(n, 3, dtype=torch.float64, device=dev)
        U = torch.empty(1, dtype=torch.float64, device=dev)
        M.mstar_accelerations_noalloc(n, torch.from_numpy(m).to(dev), torch.from_numpy(np.ascontiguousarray(r)).to(dev),
                                      1.0, a, U, torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        check(a.cpu().numpy(), float(U.item()), m, r)


def step_time(m, r, H):
    """Physical time of one step with two divisions (2 and 4 substeps), in long double, from rest."""
    m, r = m.astype(LD), r.astype(LD)
    r = r - (m[:, None] * r).sum(0) / m.sum()
    B = forces(m, r)[2]
    ts = []
    for nk in (2, 4):
        delta = LD(H) / nk
        f = delta / 2 / B
        x, v, t = r.copy(), np.zeros_like(r), f
        for tau in range(1, nk + 1):
            a, _, U = forces(m, x)
            v = v + delta / U * a
            T = (m[:, None] * v * v).sum() / 2
            f = (delta / 2 if tau == nk else delta) / (T + B)
            x = x + f * v
            t = t + f
        ts.append(t)
    return 4 * ts[1] / 3 - ts[0] / 3


@pytest.mark.parametrize("ratio", [1e4, 1e8, 1e12, 1e18])
def test_batched_sums(ratio):
    systems, H = [], []
    for n in (24, 32, 64, 65, 96):
        for place in places(n):
            m, r = system(n, ratio, place)
            d = np.sqrt(((r[:, None] - r[None]) ** 2).sum(-1)) + 1e30 * np.eye(n)
            t_dyn = np.sqrt(d.min() ** 3 / m.sum())
            systems.append((m, r, np.zeros_like(r)))
            H.append(1e-4 * t_dyn * float(forces(m, r)[2]))
    b = M.Batch(systems, eta_gbs=1e-9, k_fix=2)
    b.set_H(np.array(H))
    first = {}  # time after the first accepted attempt; each rejected one halves H
    for tries in range(30):
        b.step(1e6, 1)
        t = b.state()["t"]
        for k in range(len(systems)):
            if t[k] > 0.0 and k not in first:
                first[k] = (t[k], 0.5 ** tries)
    b.close()
    for k, (m, r, _) in enumerate(systems):
        tk, f = first[k]
        te = step_time(m, r, H[k] * f)
        assert abs(tk - te) <= 128 * U53 * te, (len(m), float(abs(tk - te) / te / U53))
