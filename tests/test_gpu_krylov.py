"""The operator passes of the FP32-V-cycle form: their FP64 sums of FP32 neighbours against numpy."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle as o  # noqa: E402
from paper_1312_2880_gb300 import hz, inputs as I  # noqa: E402


@pytest.mark.parametrize("decades", [0, 9, 18])
@pytest.mark.parametrize("n", [8, 18, 62, 128])
def test_first_step_scalars_with_wide_ranges(n, decades):
    """alpha of the first iteration is <r^, b h^2> / <r^, A y> with y the FP32 V-cycle of b, which the
    library also returns on its own. Right-hand sides spread over many decades make neighbouring y
    values differ by more than the exact FP32 addition can hold, zeros among them. Summing (n+1)^2
    products in FP64 in any order is within (n+1)^2 2^-53 of the sum of their moduli."""
    rng = np.random.default_rng(n + decades)
    m = n + 1
    b = (rng.standard_normal((m, m)) + 1j * rng.standard_normal((m, m))) * 10.0 ** rng.uniform(-decades, 0, (m, m))
    b[rng.uniform(size=(m, m)) < 0.1] = 0
    kf = I.wedge_k(n, 0.4 * n, 5)
    P = hz.Problem(n, kf, 0.5, variant="hyb", precision="fp32", levels=2 if n < 32 else 0, k_ref=0.4 * n)
    db = torch.from_numpy(b).cuda()
    y = P.vcycle(db).cpu().numpy().ravel()
    P.solve(db, tol=1e-300, maxit=1, allow_fail=True)
    s = P.krylov_scalars()
    P.close()
    h2 = 1.0 / (n * n)
    v = h2 * (o.helmholtz_matrix(n, kf) @ y)
    rh = o.shadow_residual(m * m)
    rho, rv = np.vdot(rh, h2 * b.ravel()), np.vdot(rh, v)
    bound = m * m * 2.0**-53 * (np.abs(rh) @ np.abs(h2 * b.ravel()) / abs(rho)
                                + np.abs(rh) @ (abs(h2 * o.helmholtz_matrix(n, kf)) @ np.abs(y)) / abs(rv))
    assert abs(s["alpha"] - rho / rv) <= bound * abs(rho / rv)
