"""The two-sweep tiles of large FP32 Kaczmarz levels against the colour launches."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1312_2880_gb300 import hz, inputs as I  # noqa: E402


# n_l = n / 2: 448 and 512 (tiles of 32, a remainder of one node), 768 and 832 (tiles of 64, one node) and 800
# (half a tile); two or four launches a pass, right-hand sides side by side.
@pytest.mark.parametrize("n,batch,nu", [(896, 1, 4), (896, 1, 8), (1024, 1, 4), (1536, 1, 4), (1600, 1, 8), (1664, 2, 4)])
def test_tiles_give_the_bits_of_colour_launches(n, batch, nu):
    kf = I.wedge_k(n, 0.625 * n, 11)
    rng = np.random.default_rng(n)
    rhs = torch.from_numpy(rng.standard_normal((batch, n + 1, n + 1)) + 1j * rng.standard_normal((batch, n + 1, n + 1))).cuda()
    f = torch.from_numpy(rng.standard_normal((n // 2 + 1,) * 2) + 1j * rng.standard_normal((n // 2 + 1,) * 2)).cuda()
    ec = torch.from_numpy(rng.standard_normal((n // 4 + 1,) * 2) + 1j * rng.standard_normal((n // 4 + 1,) * 2)).cuda()
    out = {}
    for form in ("tile", "colour"):
        P = hz.Problem(n, kf, 0.5, variant="hyb", precision="fp32", k_ref=0.625 * n, kacz_form=form, batch=batch, nu_kacz=nu)
        s = P.level_info(1)
        assert s["smoother"] == "kaczmarz" and s["kacz_form"] == form, s
        u, fc = P.level_presmooth(1, f)
        v = P.level_postsmooth(1, f, u, ec)
        x, _ = P.solve_batch(rhs, tol=1e-300, maxit=1, allow_fail=True)
        out[form] = [t.cpu().numpy() for t in (u, fc, v, x)]
        P.close()
    for a, b in zip(out["tile"], out["colour"]):
        assert np.array_equal(a.view(np.uint64), b.view(np.uint64))
