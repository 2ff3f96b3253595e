"""The tiled pair loop's two arithmetics (integer, and mixed FP64 / integer where a tile pair is
flat, too wide in scale or holds a very close far pair) against the oracle, body by body.

Tolerance: both sides add n terms f_ij in binary64 or better. A sum of n terms in any order errs
by at most (n - 1) u sum |f_ij| (u = 2^-53), and each term by less than 8 u of itself (separation,
1/r^3 and the product on the oracle's side; 4 u in integers), so two such sums differ by at most
2 (n + 8) u sum |f_ij| in each component, and likewise for U.
"""
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


def system(kind, n):
    m, r, v = W.plummer(n, 17)
    m, r = m.copy(), r.copy()
    u = W.Stream(17, 2).uniform(n)
    if kind == "masses":            # a mass spectrum over four decades
        m *= 10.0 ** (-4.0 * u)
    elif kind == "one_heavy":       # equal masses but for one body
        m[n // 3] *= 300.0
    elif kind == "flat":            # a thin disc: mixed arithmetic
        r[:, 2] *= 1e-6
    elif kind == "nested":          # half of the bodies in a core 1e-5 as wide
        r[n // 2:] *= 1e-5
    elif kind == "close":           # far pairs closer than 2^-10 of a tile pair's extent
        r[n // 2:] = r[:n - n // 2] + 1e-5 * (1.0 + u[n // 2:, None])
    elif kind == "apart":           # two clusters 1e4 radii apart
        r[n // 2:, 0] += 1e4
    elif kind == "tiny":            # extents below the integer window's range
        r *= 1e-12
    return m, r, v


@pytest.mark.parametrize("n,tile", [(513, 0), (544, 0), (545, 0), (577, 64), (640, 128), (641, 128)])
@pytest.mark.parametrize("kind,n_d", [("plain", 2), ("plain", 0), ("masses", 2), ("masses", 1), ("one_heavy", 2),
                                      ("flat", 2), ("nested", 2), ("close", 2), ("apart", 2), ("tiny", 2)])
def test_both_arithmetics_match_the_oracle(n, tile, kind, n_d):
    m, r, v = system(kind, n)
    g = M.Integrator(m, r, v, pair_tile=tile, n_d=n_d)
    a, U = g.accelerations()
    rs = g.state()["r"]
    g.close()
    root, par, lev, order = O.prim(rs)
    ao, Uo = O.forces(m, rs, par, lev, O.to_mst(par, rs), n_d=n_d)
    d = rs[None, :, :] - rs[:, None, :]
    dist = np.sqrt((d * d).sum(-1))
    np.fill_diagonal(dist, np.inf)
    terms = (m[None, :, None] * np.abs(d) / dist[..., None] ** 3).sum(1)
    pot = 0.5 * (m[:, None] * m[None, :] / dist).sum()
    tol = 2.0 * (n + 8) * 2.0 ** -53
    assert (np.abs(a - ao) <= tol * np.maximum(terms, 1e-300)).all(), (np.abs(a - ao) / terms).max() / tol
    assert abs(U - Uo) <= tol * pot


@pytest.mark.parametrize("n,split", [(45, 2), (200, 0), (513, 8), (900, 0)])
@pytest.mark.parametrize("n_d", [1, 2])
def test_near_pairs_of_a_node_of_high_degree(n, split, n_d):
    """A body with 12 tree neighbours (the centre of an icosahedron, whose edges are 5 % longer than
    its radius), some with children of their own: more partners than share lanes. Same tolerance."""
    m, r, v = W.plummer(n, 17)
    r = r + 20.0
    g = (1.0 + 5.0 ** 0.5) / 2.0
    ico = np.array([(0, a, b * g) for a in (-1, 1) for b in (-1, 1)], float)
    ico = np.concatenate([ico, ico[:, [1, 2, 0]], ico[:, [2, 0, 1]]]) * (1.0 + 1e-3 * np.arange(12))[:, None]
    r[0] = 0.0
    r[1:13] = ico
    r[13:25] = 1.4 * ico
    r[25:34] = 1.5 * ico[:9] + 0.1
    it = M.Integrator(m, r, v, n_d=n_d, pair_split=split)
    a, U = it.accelerations()
    rs = it.state()["r"]
    it.close()
    root, par, lev, order = O.prim(rs)
    deg = np.bincount(par[par >= 0], minlength=n) + (par >= 0)
    assert deg.max() >= 12
    ao, Uo = O.forces(m, rs, par, lev, O.to_mst(par, rs), n_d=n_d)
    d = rs[None, :, :] - rs[:, None, :]
    dist = np.sqrt((d * d).sum(-1))
    np.fill_diagonal(dist, np.inf)
    terms = (m[None, :, None] * np.abs(d) / dist[..., None] ** 3).sum(1)
    pot = 0.5 * (m[:, None] * m[None, :] / dist).sum()
    tol = 2.0 * (n + 8) * 2.0 ** -53
    # both sides take near separations from the same kind of path sums; their own rounding (3 sums of
    # coordinates below 50 over distances above 0.1) is not the oracle's: 3 * 500 u on each term
    tol += 2 * 3 * 500 * 2.0 ** -53
    assert (np.abs(a - ao) <= tol * np.maximum(terms, 1e-300)).all(), (np.abs(a - ao) / terms).max() / tol
    assert abs(U - Uo) <= tol * pot


def test_a_coincident_far_pair_is_undefined():
    """Two coincident bodies that are not tree neighbours: U and both accelerations are NaN, the
    others finite, as in the mixed arithmetic alone."""
    m, r, v = W.plummer(600, 17)
    r = r.copy()
    # a chain of bodies at the coincident point keeps the pair more than two edges apart
    r[100] = r[400]
    g = M.Integrator(m, r, v, n_d=0)
    a, U = g.accelerations()
    g.close()
    bad = np.isnan(a).any(axis=1)
    assert np.isnan(U) and bad[100] and bad[400] and bad.sum() == 2
