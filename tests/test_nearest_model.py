"""A model of the nearest-neighbour filter of csrc/nearest.cuh (float distances, then exact ones for
the undecided): whenever it calls the float nearest certain, that candidate has the strictly
smallest FP64 distance, and its limit never excludes the FP64 nearest. CPU only.

Float fused multiply-adds are modelled by one rounding of the binary64 value (the products of two
floats are exact in binary64, and a sum's rounding there is 2^-53: far below the margins).
"""
import numpy as np
import pytest

f32 = np.float32
INF = f32(np.inf)


def scan(xi, X):
    """m1, m2, j1 and e as the kernel forms them, and the FP64 distances of the CPU definition."""
    fi, F = xi.astype(f32), X.astype(f32)
    d = (fi[None, :] - F).astype(f32).astype(np.float64)
    r2 = (d[:, 0] * d[:, 0]).astype(f32).astype(np.float64)
    r2 = (d[:, 1] * d[:, 1] + r2).astype(f32).astype(np.float64)
    with np.errstate(over="ignore"):
        r2 = np.minimum((d[:, 2] * d[:, 2] + r2).astype(f32), f32(3e38))
    o = np.argsort(r2, kind="stable")
    err = lambda v: np.abs(v.astype(f32)).max(axis=-1) * f32(2.0 ** -23) + f32(1e-37)  # noqa: E731
    e = f32(err(xi) + err(X).max())
    dd = xi[None, :] - X
    exact = (dd[:, 0] * dd[:, 0] + dd[:, 1] * dd[:, 1]) + dd[:, 2] * dd[:, 2]
    return r2, r2[o[0]], r2[o[1]], o[0], e, exact


def certain(m1, m2, e):
    s1, s2 = np.sqrt(m1), np.sqrt(m2)
    return 1e-30 < m1 < 1e30 and s2 * f32(1 - 2.0 ** -18) - f32(1.75) * e > s1 * f32(1 + 2.0 ** -18) + f32(1.75) * e


def limit(m1, e):
    if not m1 < 1e30:
        return INF
    t = np.sqrt(max(m1, f32(1e-30))) * f32(1 + 2.0 ** -17) + f32(3.75) * e
    return t * t * f32(1 + 2.0 ** -16)


@pytest.mark.parametrize("scale", [1e-14, 1e-3, 1.0, 1e4, 1e12])
@pytest.mark.parametrize("offset", [0.0, 1.0, 1e3, 1e6])
@pytest.mark.parametrize("gap", [0.0, 1e-9, 1e-7, 1e-6, 1e-4])
def test_filter_decides_as_fp64(scale, offset, gap):
    rng = np.random.default_rng(int(1e6 * gap * 1e3 + offset) % (1 << 30) + 17)
    sure = 0
    for _ in range(200):
        xi = scale * (offset * rng.uniform(-1, 1, 3) + rng.uniform(-1, 1, 3))
        # candidates at nearly one distance from xi, differing by the relative gap
        u = rng.normal(size=(6, 3))
        u /= np.linalg.norm(u, axis=1)[:, None]
        rad = scale * rng.uniform(0.01, 1.0) * (1.0 + gap * rng.uniform(-1, 1, 6))
        X = xi + rad[:, None] * u
        r2, m1, m2, j1, e, exact = scan(xi, X)
        best = exact.min()
        if certain(m1, m2, e):
            sure += 1
            assert exact[j1] == best and (exact == best).sum() == 1
        lim = limit(m1, e)
        assert (r2[exact == best] <= lim).all()
    if gap >= 1e-4 and offset <= 1.0 and scale > 1e-13:
        assert sure > 100  # the filter is of use
