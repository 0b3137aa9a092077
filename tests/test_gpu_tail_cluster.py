"""The FP64 coarse tail whose coarsest solve is shared by a cluster, against the levels run one by one."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1312_2880_gb300 import hz, inputs as I  # noqa: E402


# Coarsest grids of (nc + 1)^2 = 16 (one block), 25 .. 81 unknowns: a ragged last share, shares beyond
# the last row (25 and 36 rows over eight blocks), the largest coarsest grid of an FP64 tail. 19 instances
# are the last batch on clusters on 152 SMs, 20 the first on single blocks.
@pytest.mark.parametrize("nc", [3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("batch", [1, 3, 19, 20])
def test_tail_gives_the_bits_of_the_levels(nc, batch):
    n = 4 * nc
    kf = I.wedge_k(n, 0.3 * n, 11)
    rng = np.random.default_rng(n)
    rhs = torch.from_numpy(rng.standard_normal((batch, n + 1, n + 1)) + 1j * rng.standard_normal((batch, n + 1, n + 1))).cuda()
    out = []
    for tail in (True, False):
        P = hz.Problem(n, kf, 0.5, variant="hyb", precision="fp64", k_ref=0.3 * n, coarse_tail=tail, batch=batch, levels=3)
        assert any(d["in_tail"] for d in P.schedule()) == tail, P.schedule()
        z = P.vcycle(rhs[0].contiguous())
        x, _ = P.solve_batch(rhs, tol=1e-300, maxit=2, allow_fail=True)
        out.append([t.cpu().numpy() for t in (z, x)])
        P.close()
    for a, b in zip(*out):
        assert np.array_equal(a.view(np.uint64), b.view(np.uint64))
