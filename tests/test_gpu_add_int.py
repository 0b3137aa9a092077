"""Sums formed on the integer pipe: the operator on fields whose neighbours differ by any exponent."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1312_2880_gb300 import hz, inputs as I  # noqa: E402


@pytest.mark.parametrize("case", ["wide", "near", "cancel", "sparse", "tiny", "huge", "special"])
def test_operator_neighbour_sums_are_correctly_rounded(case):
    """n = 512 takes the integer additions. (W + E) + (S + N), k = 0 diagonal -4 and the scale n^2 = 2^18
    leave v = 2^18 (nb - 4 u) with one rounding in each step, as numpy does them; interior nodes."""
    n = 512
    rng = np.random.default_rng(len(case))
    m = n + 1
    re = lambda: rng.standard_normal((m, m))
    u = re() + 1j * re()
    if case == "wide":
        u = u * 2.0 ** rng.integers(-70, 70, (m, m))
    elif case == "near":  # few significant bits: ties and carries
        u = (rng.integers(-8, 9, (m, m)) * 2.0 ** rng.integers(0, 55, (m, m))) + 1j * rng.integers(-3, 4, (m, m))
    elif case == "cancel":  # neighbours nearly opposite
        s = np.where((np.indices((m, m)).sum(0) // 2) % 2, 1.0, -1.0)
        u = s * (1.0 + 2.0**-50 * rng.integers(-4, 5, (m, m))) + 1j * s * (3.0 + 2.0**-45 * re())
    elif case == "sparse":
        u = np.where(rng.uniform(size=(m, m)) < 0.5, u, 0) * np.where(rng.uniform(size=(m, m)) < 0.5, 1.0, -1.0)
    elif case == "tiny":  # subnormal sums
        u = u * 2.0 ** rng.integers(-1074, -1000, (m, m))
    elif case == "huge":
        u = u * 2.0 ** rng.integers(960, 1000, (m, m))
    elif case == "special":
        u[rng.uniform(size=(m, m)) < 0.01] = np.inf
        u[rng.uniform(size=(m, m)) < 0.01] = np.nan
    P = hz.Problem(n, np.full((m, m), 1e-30), 0.5, k_ref=1.0, variant="sl_plain")
    v = P.apply(torch.from_numpy(u).cuda()).cpu().numpy()[1:-1, 1:-1]
    P.close()
    with np.errstate(all="ignore"):
        for part in ("real", "imag"):
            a = getattr(u, part)
            nb = (a[1:-1, :-2] + a[1:-1, 2:]) + (a[:-2, 1:-1] + a[2:, 1:-1])
            c = a[1:-1, 1:-1]
            # fma(-4, c, nb): -4 c is exact, so one rounding
            ref = (nb + -4.0 * c) * float(n * n)
            got = getattr(v, part)
            assert np.array_equal(got, ref, equal_nan=True)
