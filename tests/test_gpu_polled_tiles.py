"""Non-blocking solves, whose Kaczmarz tiles differ from the blocking ones', against them and beside each other."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1312_2880_gb300 import hz, inputs as I  # noqa: E402


@pytest.mark.parametrize("nu", [4, 8])
def test_polled_solves_keep_the_bits_of_blocking_ones(nu):
    """n_l = 128 takes four-sweep tiles in a blocking solve: one launch a pass (four sweeps) that ends in the other
    array, against two that end in their own. Blocking, polled and blocking again on one problem."""
    n = 256
    kf = I.grf_k(n, 0.5 * n, 7)
    rng = np.random.default_rng(nu)
    b = torch.from_numpy(rng.standard_normal((n + 1, n + 1)) + 1j * rng.standard_normal((n + 1, n + 1))).cuda()
    for tail in (True, False):
        P = [hz.Problem(n, kf, 0.5, precision="fp32", k_ref=0.5 * n, nu_kacz=nu, coarse_tail=tail) for _ in range(3)]
        assert any(d["kacz_form"] == "tile" for d in P[0].schedule()), P[0].schedule()
        ref, info, hist = P[0].solve(b, tol=1e-14, maxit=4, allow_fail=True)
        z = P[0].vcycle(b)
        xs = [torch.empty_like(b) for _ in P]
        for p, x in zip(P, xs):
            p.solve_start(b, x, tol=1e-14, maxit=4)
        for p, x in zip(P, xs):
            _, i2, h2 = p.solve_finish(allow_fail=True)
            assert torch.equal(torch.view_as_real(x), torch.view_as_real(ref))
            assert i2["iterations"] == info["iterations"] and np.array_equal(h2, hist)
        again, _, _ = P[1].solve(b, tol=1e-14, maxit=4, allow_fail=True)
        assert torch.equal(torch.view_as_real(again), torch.view_as_real(ref))
        assert torch.equal(torch.view_as_real(P[1].vcycle(b)), torch.view_as_real(z))
        for p in P:
            p.close()
