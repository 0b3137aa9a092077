"""The one-launch Kaczmarz passes (tiles with the halo of all four sweeps) against the colour launches."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1312_2880_gb300 import hz, inputs as I  # noqa: E402


# Level sizes n_l = n / 2 around multiples of the tile sizes 13, 37 and 62 (n_l + 1 nodes a side), a
# level smaller than one tile, several tiles with a remainder of one node, and levels wide enough
# for tiles without a boundary row. Batches move the choice of the tile, sweep counts the number
# of launches (one to three).
@pytest.mark.parametrize("n", [20, 64, 68, 88, 92, 136, 200, 288, 352, 640])
@pytest.mark.parametrize("batch,nu", [(1, 4), (3, 4), (16, 4), (1, 2), (1, 6), (1, 8)])
def test_pass_gives_the_bits_of_colour_launches(n, batch, nu):
    kf = I.wedge_k(n, 0.625 * n, 11)
    rng = np.random.default_rng(n)
    rhs = rng.standard_normal((batch, n + 1, n + 1)) + 1j * rng.standard_normal((batch, n + 1, n + 1))
    f = torch.from_numpy(rng.standard_normal((n // 2 + 1,) * 2) + 1j * rng.standard_normal((n // 2 + 1,) * 2)).cuda()
    ec = torch.from_numpy(rng.standard_normal((n // 4 + 1,) * 2) + 1j * rng.standard_normal((n // 4 + 1,) * 2)).cuda()
    out = {}
    for form in ("tile", "colour"):
        P = hz.Problem(n, kf, 0.5, variant="hyb", precision="fp32", levels=3 if n < 128 else 0, k_ref=0.625 * n,
                       coarse_tail=False, kacz_form=form, batch=batch, nu_kacz=nu)
        s = P.level_info(1)
        assert s["smoother"] == "kaczmarz" and s["kacz_form"] == form, s
        u, fc = P.level_presmooth(1, f)
        v = P.level_postsmooth(1, f, u, ec)
        x, _ = P.solve_batch(torch.from_numpy(rhs).cuda(), tol=1e-300, maxit=2, allow_fail=True)
        out[form] = [t.cpu().numpy() for t in (u, fc, v, x)]
        P.close()
    for a, b in zip(out["tile"], out["colour"]):
        assert np.array_equal(a.view(np.uint64), b.view(np.uint64))
