"""The pair loops at the ends of the integer arithmetic's range of masses and lengths, where m / r^2
falls below the smallest normal float: forces against long double sums.

Tolerance (u = 2^-53), relative to the sum of the terms' magnitudes: a term errs by 4 u (positions
rounded by 2^-53 of r, three roundings in m d / r^3), the 32 terms that a warp adds in integers by 2 u
of their sum, and the binary64 additions after that form chains of at most 8 (warps), 4 (slots), 4
(flush, G, finish): 22 u, and 24 u is taken.
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


def shell(n, radius, mass):
    """Bodies on a sphere, masses alike but not equal."""
    s = W.Stream(37, n)
    x = np.stack([s.uniform(n) - 0.5 for _ in range(3)], 1)
    x *= (radius / np.linalg.norm(x, axis=1))[:, None]
    return mass * (1.0 + 0.05 * s.uniform(n)), x


def check(a, m, r):
    m, r = m.astype(np.longdouble), r.astype(np.longdouble)
    d = r[None] - r[:, None]
    r2 = (d * d).sum(-1)
    np.fill_diagonal(r2, 1)
    w = m[None] / (r2 * np.sqrt(r2))
    np.fill_diagonal(w, 0)
    err = np.abs(a - (w[..., None] * d).sum(1)).max(1)
    bound = (w * np.sqrt(r2)).sum(1)
    assert (err <= 24 * 2.0 ** -53 * bound).all(), float((err / bound).max() * 2.0 ** 53)


@pytest.mark.parametrize("radius,mass", [(9.9e14, 9.3e-13), (1e14, 1e-12), (9.9e14, 1e-6), (9.9e14, 1.0), (1e-8, 1e12)])
@pytest.mark.parametrize("n", [32, 64, 100])
def test_forces(n, radius, mass):
    m, r = shell(n, radius, mass)
    dev = torch.device("cuda")
    a = torch.empty(n, 3, dtype=torch.float64, device=dev)
    U = torch.empty(1, dtype=torch.float64, device=dev)
    M.mstar_accelerations_noalloc(n, torch.from_numpy(m).to(dev), torch.from_numpy(r).to(dev), 1.0, a, U,
                                  torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    check(a.cpu().numpy(), m, r)
    g = M.Integrator(m, r, np.zeros_like(r), n_d=0)
    ac, _ = g.accelerations()
    rs = g.state()["r"]
    g.close()
    check(ac, m, rs)
