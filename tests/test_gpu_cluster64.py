"""The FP64 cluster form of a Kaczmarz level against the colour launches: bands of two rows and more, a
last band of one row, empty blocks, one and two lanes per row action, 1024-thread blocks."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1312_2880_gb300 import hz, inputs as I  # noqa: E402


# n_l = n / 2: 16 (two rows a band, the last with one), 18, 30, 32 (three rows, empty blocks), 48, 60, 64,
# 96, 120, 128, 144 and 208 (more than 256 blocks of five nodes a band)
@pytest.mark.parametrize("nl", [16, 18, 30, 32, 48, 60, 64, 96, 120, 128, 144, 208])
@pytest.mark.parametrize("batch", [1, 2])
def test_cluster_gives_the_bits_of_colour_launches(nl, batch):
    n = 2 * nl
    kf = I.wedge_k(n, 0.625 * n, 11)
    rng = np.random.default_rng(n)
    c = lambda *s: torch.from_numpy(rng.standard_normal(s) + 1j * rng.standard_normal(s)).cuda()
    rhs, f, ec = c(batch, n + 1, n + 1), c(nl + 1, nl + 1), c(nl // 2 + 1, nl // 2 + 1)
    out = {}
    for form in ("cluster", "colour"):
        P = hz.Problem(n, kf, 0.5, variant="hyb", levels=3 if n < 128 else 0, k_ref=0.625 * n, coarse_tail=False,
                       kacz_form=form, batch=batch)
        s = P.level_info(1)
        assert s["smoother"] == "kaczmarz" and s["kacz_form"] == form, s
        u, fc = P.level_presmooth(1, f)
        v = P.level_postsmooth(1, f, u, ec)
        x, _ = P.solve_batch(rhs, tol=1e-300, maxit=2, allow_fail=True)
        out[form] = [t.cpu().numpy() for t in (u, fc, v, x)]
        P.close()
    for a, b in zip(out["cluster"], out["colour"]):
        assert np.array_equal(a.view(np.uint64), b.view(np.uint64))
