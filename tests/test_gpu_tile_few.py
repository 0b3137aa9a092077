"""The fused FP64 passes on small levels (16 x 4 tiles, one block per SM at most) against the streaming form."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1312_2880_gb300 import hz, inputs as I  # noqa: E402


# Grids within one tile, whole tiles and one node more, ragged last tiles; the last size of the small
# tiles on 152 SMs (6 x 24 of them at n = 92, 7 x 25 at 96); batches that move that limit; every
# operator pair (complex, real or mixed diagonals).
@pytest.mark.parametrize("n", [8, 12, 16, 32, 40, 60, 64, 88, 92, 96, 112])
@pytest.mark.parametrize("variant", ["hyb", "sl", "sl_plain"])
@pytest.mark.parametrize("batch", [1, 5])
def test_small_levels_give_the_bits_of_the_streaming_form(n, variant, batch):
    kf = I.wedge_k(n, 0.3 * n, 11)
    rng = np.random.default_rng(n)
    rhs = torch.from_numpy(rng.standard_normal((batch, n + 1, n + 1)) + 1j * rng.standard_normal((batch, n + 1, n + 1))).cuda()
    out = []
    for form in (0, 1):
        P = hz.Problem(n, kf, 0.5, variant=variant, precision="fp64", k_ref=0.3 * n, coarse_tail=False, batch=batch,
                       levels=2 if n <= 64 else 3, pass_variant=form)
        s = P.level_info(0)
        assert s["smoother"] == "gs" and s["pass_down"] == form, s
        z = P.vcycle(rhs[0].contiguous())
        x, _ = P.solve_batch(rhs, tol=1e-300, maxit=2, allow_fail=True)
        out.append([t.cpu().numpy() for t in (z, x)])
        P.close()
    for a, b in zip(*out):
        assert np.array_equal(a.view(np.uint64), b.view(np.uint64))
