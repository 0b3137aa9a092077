"""The coarsest solve over several blocks: sizes around its row groups and column chunks."""
import numpy as np
import pytest

import oracle as o

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1312_2880_gb300 import hz, inputs as I  # noqa: E402


# Coarsest grids of (n_c + 1)^2 = 9 .. 1089 unknowns: less than one group of 16 rows, one column chunk
# (48 columns in FP64, 112 in FP32) and its neighbours, and the largest the library takes.
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("nc", [2, 3, 6, 9, 10, 15, 16, 27, 31, 32])
def test_coarse_solve(nc, precision):
    n, k = 4 * nc, 1.3 * nc
    kf = I.wedge_k(n, k, 3)
    P = hz.Problem(n, kf, 0.5, variant="hyb", precision=precision, levels=3, k_ref=k)
    rng = np.random.default_rng(nc)
    f = rng.standard_normal((nc + 1, nc + 1)) + 1j * rng.standard_normal((nc + 1, nc + 1))
    u = P.coarse_solve(torch.from_numpy(f).cuda()).cpu().numpy().ravel()
    P.close()
    A = o.helmholtz_matrix(nc, kf[::4, ::4]).toarray()
    ref = np.linalg.solve(A, f.ravel())
    # |A^-1| |A| amplifies the rounding of the inverse and of the sums of m products
    m = (nc + 1) ** 2
    bound = 4 * m * np.linalg.cond(A) * (2.0**-53 if precision == "fp64" else 2.0**-24)
    assert np.linalg.norm(u - ref) <= min(bound, 0.1) * np.linalg.norm(ref)


def test_coarse_solve_in_a_batch():
    """Every right-hand side of a batch takes its own coarsest level (the bits of single solves)."""
    n = 124  # coarsest 31: 1024 unknowns
    kf = I.constant_k(n, 0.4 * n)
    rhs = np.stack([I.point_source_rhs(n, I.random_interior_nodes(n, 2, s)) for s in (4, 5, 6)])
    P = hz.Problem(n, kf, 0.5, precision="fp32", k_ref=0.4 * n, batch=3)
    xb = P.solve_batch(torch.from_numpy(rhs).cuda(), tol=1e-300, maxit=3, allow_fail=True)[0].cpu().numpy()
    P.close()
    S = hz.Problem(n, kf, 0.5, precision="fp32", k_ref=0.4 * n)
    for q in range(3):
        x = S.solve(torch.from_numpy(rhs[q]).cuda(), tol=1e-300, maxit=3, allow_fail=True)[0].cpu().numpy()
        assert np.array_equal(x.view(np.uint64), xb[q].view(np.uint64))
    S.close()
