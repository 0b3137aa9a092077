"""FP64 Kaczmarz sweeps in halo tiles of 16 to 44 nodes against the colour launches, and the default form."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1312_2880_gb300 import hz, inputs as I  # noqa: E402


# n_l = n / 2, n_l + 1 nodes a side. One instance: levels smaller than a tile, whole tiles and one node
# more, and about the last level of each edge's range and the first of the next (12 tiles a side at most
# on 152 SMs: 16 up to n_l = 190, then 192, 240, 288, 336, 432 and 528; the coarsest grid has to be
# small, which leaves these). Batches move the choice of the edge.
@pytest.mark.parametrize("n,batch", [(12, 1), (28, 1), (64, 1), (320, 1), (352, 1), (368, 1), (384, 1), (464, 1),
                                     (480, 1), (544, 1), (576, 1), (640, 1), (672, 1), (832, 1), (864, 1), (1024, 1),
                                     (1088, 1), (64, 3), (96, 3), (192, 3), (320, 2), (44, 16), (112, 16)])
def test_tiles_give_the_bits_of_colour_launches(n, batch):
    kf = I.wedge_k(n, 0.625 * n, 11)
    rng = np.random.default_rng(n)
    rhs = rng.standard_normal((batch, n + 1, n + 1)) + 1j * rng.standard_normal((batch, n + 1, n + 1))
    f = torch.from_numpy(rng.standard_normal((n // 2 + 1,) * 2) + 1j * rng.standard_normal((n // 2 + 1,) * 2)).cuda()
    ec = torch.from_numpy(rng.standard_normal((n // 4 + 1,) * 2) + 1j * rng.standard_normal((n // 4 + 1,) * 2)).cuda()
    out = {}
    for form in ("tile", "colour"):
        P = hz.Problem(n, kf, 0.5, variant="hyb", precision="fp64", levels=3 if n < 128 else 0, k_ref=0.625 * n, coarse_tail=False,
                       kacz_form=form, batch=batch)
        s = P.level_info(1)
        assert s["smoother"] == "kaczmarz" and s["kacz_form"] == form, s
        u, fc = P.level_presmooth(1, f)
        v = P.level_postsmooth(1, f, u, ec)
        x, _ = P.solve_batch(torch.from_numpy(rhs).cuda(), tol=1e-300, maxit=2, allow_fail=True)
        out[form] = [t.cpu().numpy() for t in (u, fc, v, x)]
        P.close()
    for a, b in zip(out["tile"], out["colour"]):
        assert np.array_equal(a.view(np.uint64), b.view(np.uint64))


@pytest.mark.parametrize("n,batch,form", [(288, 1, "cluster"), (304, 1, "tile"), (448, 1, "tile"), (448, 2, "cluster"),
                                          (1024, 2, "tile"), (1536, 1, "tile"), (1600, 1, "colour")])
def test_default_form_of_an_fp64_level(n, batch, form):
    P = hz.Problem(n, I.wedge_k(n, 0.625 * n, 11), 0.5, variant="hyb", precision="fp64", k_ref=0.625 * n, batch=batch)
    s = P.level_info(1)
    P.close()
    assert s["smoother"] == "kaczmarz" and s["kacz_form"] == form, s
