"""The two-sided block elimination of the ray problem at small and odd numbers of ray rows."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1312_2880_gb300 import hz, inputs as I  # noqa: E402


# Ray rows Nr = cells + 1: one row below the middle and none above it (Nr = 2), one on each side (3),
# unequal sides (4, 6), and a block row wider than the elements a warp fetches ahead (Nr = 73, Bs = 584).
@pytest.mark.parametrize("n,m", [(16, 16), (16, 8), (12, 4), (16, 4), (20, 4), (32, 4), (36, 4), (288, 4)])
def test_solve_has_a_small_backward_error(n, m):
    """|g - A z| against |A| |z| + |g|: these small ray grids are ill-conditioned (nearly dependent
    plane waves), so the residual is measured as a backward error; 1e-11 is the residual bound of
    the well-conditioned grids (test_gpu_ray)."""
    k = 2.3 / m * n  # k H = 2.3
    P = hz.Problem(n, I.constant_k(n, k), 0.5, variant="hlm", levels=2 if n <= 36 else 0, k_ref=k)
    R = hz.Ray(P, k, m)
    Nr, Bs = R.nc + 1, 8 * (R.nc + 1)
    assert Nr == n // m + 1
    Lb, Db, Ub = (t.cpu().numpy() for t in R.blocks())
    rng = np.random.default_rng(n + m)
    g = rng.standard_normal(R.unknowns) + 1j * rng.standard_normal(R.unknowns)
    z = R.coarse_solve(torch.from_numpy(g).cuda()).cpu().numpy().reshape(Nr, Bs)
    r = g.reshape(Nr, Bs) - np.einsum("jab,jb->ja", Db, z)
    r[1:] -= np.einsum("jab,jb->ja", Lb[1:], z[:-1])
    r[:-1] -= np.einsum("jab,jb->ja", Ub[:-1], z[1:])
    R.close()
    P.close()
    norm = np.sqrt(sum((np.abs(b) ** 2).sum() for b in (Lb, Db, Ub)))
    assert np.linalg.norm(r) <= 1e-11 * (norm * np.linalg.norm(z) + np.linalg.norm(g))
