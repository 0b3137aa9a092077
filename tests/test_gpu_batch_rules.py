"""Rules that count a batch's right-hand sides: which levels the FP64 coarse tail takes, and the operator's sums."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1312_2880_gb300 import hz, inputs as I  # noqa: E402


def _tail(n, kh, **opts):
    P = hz.Problem(n, I.grf_k(n, kh * n, 7), 0.5, k_ref=kh * n, **opts)
    s = P.schedule()
    P.close()
    return [d["n"] for d in s if d["in_tail"]]


def test_tail_levels_of_batches_and_of_given_forms():
    """On 152 SMs: 16 intervals alone, 32 from 39 right-hand sides, 48 from 61, and from there any coarsest grid (100
    unknowns below; FP32 256); Kaczmarz levels of a given form other than the default ones wherever they fit."""
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the limits are stated for 152 SMs")
    for batch, want in ((1, [16, 8]), (38, [16, 8]), (39, [32, 16, 8]), (152, [32, 16, 8])):
        assert _tail(64, 0.55, batch=batch) == want, batch
    assert _tail(96, 0.3125, batch=60) == [24, 12, 6]
    assert _tail(96, 0.3125, batch=61) == [48, 24, 12, 6]
    assert _tail(88, 0.3125, batch=60) == [] and _tail(88, 0.3125, batch=61) == [44, 22, 11]  # 144 unknowns
    assert _tail(136, 0.3125, batch=60, precision="fp32") == [] != _tail(136, 0.3125, batch=61, precision="fp32")
    for form in ("colour", "grid", "level"):
        assert _tail(128, 0.4, kacz_form=form) == [32, 16, 8], form
    assert _tail(128, 0.4) == [16, 8]
    assert _tail(128, 0.08, pass_variant=5) == _tail(128, 0.08, pass_variant=0) == [16, 8]  # the passes' form does not move it


@pytest.mark.parametrize("n,batch", [(64, 39), (88, 61), (96, 61), (128, 15), (128, 16)])
def test_batches_keep_the_bits_of_single_solves(n, batch):
    """Batches on either side of the limits: the tail's levels, its clusters (15 and 16 instances), the operator's sums."""
    kf = I.grf_k(n, 0.55 * n, 7)
    rng = np.random.default_rng(n + batch)
    rhs = torch.from_numpy(rng.standard_normal((batch, n + 1, n + 1)) + 1j * rng.standard_normal((batch, n + 1, n + 1))).cuda()
    P = hz.Problem(n, kf, 0.5, precision="fp64", k_ref=0.55 * n, batch=batch)
    xb, _ = P.solve_batch(rhs, tol=1e-300, maxit=3, allow_fail=True)
    P.close()
    S = hz.Problem(n, kf, 0.5, precision="fp64", k_ref=0.55 * n, coarse_tail=False)
    for q in (0, batch // 2, batch - 1):
        x, _, _ = S.solve(rhs[q].contiguous(), tol=1e-300, maxit=3, allow_fail=True)
        assert torch.equal(torch.view_as_real(x), torch.view_as_real(xb[q])), q
    S.close()
