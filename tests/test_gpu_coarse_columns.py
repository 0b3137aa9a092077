"""The coarsest solve column by column: a right-hand side of one node gives one column of the inverse."""
import numpy as np
import pytest

import oracle as o

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1312_2880_gb300 import hz, inputs as I  # noqa: E402


@pytest.mark.parametrize("precision,chunk", [("fp64", 48), ("fp32", 112)])
@pytest.mark.parametrize("nc", [2, 6, 10, 15, 27, 31, 32])
def test_one_node_gives_one_column(nc, precision, chunk):
    """Columns at the edges of the chunks the products are formed in, and the last one. Every other product is an
    exact zero, so u is one entry of the inverse times f: three roundings (the entry, f h^2 and their product) and
    the error of the FP64 inverse. The FP32 form's operator is that of k H in FP32 (its levels hold k H so)."""
    n, k = 4 * nc, 1.3 * nc
    kf = I.wedge_k(n, k, 3)
    m = (nc + 1) ** 2
    kH = (kf * (1.0 / n))[::4, ::4] * 4
    if precision == "fp32":
        kH = kH.astype(np.float32).astype(np.float64)
    A = o.helmholtz_matrix(nc, kH * nc).toarray()
    inv = np.linalg.inv(A)
    eps = 2.0**-53 if precision == "fp64" else 2.0**-24
    amplified = 4 * m * np.linalg.cond(A) * 2.0**-53
    cols = sorted({c for b in range(0, m + chunk, chunk) for c in (b - 1, b) if 0 <= c < m} | {0, m // 2, m - 1})
    P = hz.Problem(n, kf, 0.5, variant="hyb", precision=precision, levels=3, k_ref=k)
    for c in cols:
        f = np.zeros(m, dtype=np.complex128)
        f[c] = 1.0
        u = P.coarse_solve(torch.from_numpy(f.reshape(nc + 1, nc + 1)).cuda()).cpu().numpy().ravel()
        for got, ref in ((u.real, inv[:, c].real), (u.imag, inv[:, c].imag)):
            assert np.all(np.abs(got - ref) <= 4 * eps * np.abs(ref) + amplified * np.abs(inv[:, c]).max()), c
    P.close()
