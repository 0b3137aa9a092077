"""The FP64 restricted residual by blocks of 16 x 4 coarse nodes against the whole-level form's own restriction."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1312_2880_gb300 import hz, inputs as I  # noqa: E402


# Level sizes n_l = n / 2 with n_l / 2 + 1 coarse nodes a side: fewer than a block, whole blocks, one
# node more, ragged in both directions; one and several instances.
@pytest.mark.parametrize("n", [12, 24, 28, 44, 56, 60, 64, 68, 120, 128, 192])
@pytest.mark.parametrize("batch", [1, 3])
def test_restricted_residual_has_the_bits_of_the_cluster_form(n, batch):
    kf = I.wedge_k(n, 0.625 * n, 11)
    rng = np.random.default_rng(n)
    rhs = torch.from_numpy(rng.standard_normal((batch, n + 1, n + 1)) + 1j * rng.standard_normal((batch, n + 1, n + 1))).cuda()
    f = torch.from_numpy(rng.standard_normal((n // 2 + 1,) * 2) + 1j * rng.standard_normal((n // 2 + 1,) * 2)).cuda()
    out = []
    for form in ("tile", "cluster"):
        P = hz.Problem(n, kf, 0.5, variant="hyb", precision="fp64", levels=3 if n < 128 else 0, k_ref=0.625 * n,
                       coarse_tail=False, kacz_form=form, batch=batch)
        s = P.level_info(1)
        assert s["smoother"] == "kaczmarz" and s["kacz_form"] == form, s
        u, fc = P.level_presmooth(1, f)
        x, _ = P.solve_batch(rhs, tol=1e-300, maxit=2, allow_fail=True)
        out.append([t.cpu().numpy() for t in (u, fc, x)])
        P.close()
    for a, b in zip(*out):
        assert np.array_equal(a.view(np.uint64), b.view(np.uint64))
