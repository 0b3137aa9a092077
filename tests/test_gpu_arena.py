"""Vectors that share a place in the arena: the finest correction with t, the true residual with s."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1312_2880_gb300 import hz, inputs as I  # noqa: E402


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("tol,maxit", [(1e-6, 100), (1e-18, 60)])
def test_batch_instances_that_stop_and_restart_apart_keep_the_bits_of_single_solves(precision, tol, maxit):
    """n = 36: the arrays' pitches differ (37 and 64), so instances of the shared vectors overlap in different
    places. Right-hand sides that stop at different iterations, one that is zero, and a tolerance below the
    attainable accuracy, where every instance restarts from its true residual."""
    n, k = 36, 11.0
    kf = I.wedge_k(n, k, 3)
    rng = np.random.default_rng(5)
    rhs = np.zeros((4, n + 1, n + 1), dtype=np.complex128)
    rhs[0, n // 2, n // 3] = n * n
    rhs[1] = rng.standard_normal((n + 1, n + 1)) + 1j * rng.standard_normal((n + 1, n + 1))
    rhs[3, 2, 2] = 1j * n * n
    b = torch.from_numpy(rhs).cuda()
    P = hz.Problem(n, kf, 0.5, precision=precision, k_ref=k, batch=4)
    xb, infos = P.solve_batch(b, tol=tol, maxit=maxit, allow_fail=True)
    P.close()
    S = hz.Problem(n, kf, 0.5, precision=precision, k_ref=k)
    restarts = 0
    for q in range(4):
        x, info, _ = S.solve(b[q].contiguous(), tol=tol, maxit=maxit, allow_fail=True)
        restarts += info["restarts"]
        assert info["iterations"] == infos[q]["iterations"] and info["status"] == infos[q]["status"]
        assert torch.equal(torch.view_as_real(x), torch.view_as_real(xb[q])), q
    S.close()
    assert (restarts > 0) == (tol < 1e-10)
    assert not xb[2].any()
