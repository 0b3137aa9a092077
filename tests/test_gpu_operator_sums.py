"""Parts of the operator kernels of the FP32-V-cycle form on their own: the FP64 sum of four FP32 values without
FP64 additions, and launches whose blocks carry two blocks of the reduction."""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1312_2880_gb300 import build  # noqa: E402

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("probe") / "krylov_probe.so")
    csrc = os.path.join(os.path.dirname(HERE), "paper_1312_2880_gb300", "csrc")
    subprocess.run([build._nvcc(), "-shared", *build.ARCH, *build.FLAGS, "-I" + csrc,
                    os.path.join(HERE, "krylov_probe.cu"), "-o", so], check=True)
    return ctypes.CDLL(so)


def _ptr(t):
    return ctypes.c_void_p(t.data_ptr())


def _values(kind, count, rng):
    """(count, 4) FP32 values W, E, S, N of one component."""
    f = np.float32
    m = rng.standard_normal((count, 4)).astype(f)
    sign = np.where(rng.uniform(size=(count, 4)) < 0.5, f(1), f(-1))
    exp = lambda lo, hi: np.exp2(rng.integers(lo, hi, (count, 4)).astype(np.float64)).astype(f)
    if kind == "near":
        return m
    if kind == "wide":
        return m * exp(-60, 60)
    if kind == "powers":  # powers of two and what is far below them, of either sign
        v = sign * exp(-70, 3)
        v[:, 0] = np.abs(v[:, 0]) * 0 + 1
        return v
    if kind == "next to powers":  # leading bits that a remainder of the other sign takes away
        v = sign * exp(-30, -20) * (1 + exp(-23, 0))
        v[:, 0] = np.where(rng.uniform(size=count) < 0.5, f(1), np.nextafter(f(1), f(0)))
        return v
    if kind == "cancel":  # W + E and S + N nearly opposite, or W and E
        v = m.copy()
        v[:, 2] = -v[:, 0] * (1 + f(2.0**-23) * rng.integers(-2, 3, count).astype(f))
        v[:, 3] = np.where(rng.uniform(size=count) < 0.5, -v[:, 1], v[:, 3] * f(2.0**-30))
        return v
    if kind == "long remainders":  # 24 bits in each of up to four ranges below each other
        v = (1 + exp(-23, 0)) * sign * np.exp2(np.array([0.0, -24, -48, -72])).astype(f)
        return rng.permuted(v, axis=1)
    if kind == "sparse":
        return np.where(rng.uniform(size=(count, 4)) < 0.6, f(0), m * exp(-12, 12))
    if kind == "subnormal":
        return (rng.integers(-(1 << 24), 1 << 24, (count, 4)) * 2.0**-149).astype(f) * np.where(
            rng.uniform(size=(count, 4)) < 0.3, exp(0, 40), f(1))
    if kind == "huge":
        return (m * f(2.0**125)).clip(-3.4e38, 3.4e38).astype(f)
    v = m.copy()  # special
    v[rng.uniform(size=v.shape) < 0.3] = np.inf
    v[rng.uniform(size=v.shape) < 0.2] *= f(-1)
    v[rng.uniform(size=v.shape) < 0.2] = np.nan
    return v


KINDS = ("near", "wide", "powers", "next to powers", "cancel", "long remainders", "sparse", "subnormal", "huge", "special")


@pytest.mark.parametrize("kind", KINDS)
def test_neighbour_sum_is_exact_or_the_fp64_sum(probe, kind):
    """Where nb_sum takes a node its value is the exact sum; elsewhere the operator adds in FP64, (W + E) + (S + N),
    with subnormal FP32 values as zeros (the widening of the other FP64 kernels)."""
    rng = np.random.default_rng(KINDS.index(kind))
    count = 4000
    re, im = _values(kind, count, rng), _values(kind, count, rng)
    v = torch.from_numpy(np.stack([re, im], -1).astype(np.float32)).cuda()
    total, value = (torch.empty(count, 2, dtype=torch.float64, device="cuda") for _ in range(2))
    odd = torch.empty(count, dtype=torch.int32, device="cuda")
    assert probe.probe_nb_sum(_ptr(v), _ptr(total), _ptr(value), _ptr(odd), count) == 0
    total, value, odd = total.cpu().numpy(), value.cpu().numpy(), odd.cpu().numpy()
    for c, a in enumerate((re, im)):
        wide = np.where(np.abs(a) < 2.0**-126, 0.0, a.astype(np.float64))
        with np.errstate(all="ignore"):
            fp64 = (wide[:, 0] + wide[:, 1]) + (wide[:, 2] + wide[:, 3])
        bad = odd != 0
        assert np.array_equal(total[bad, c], fp64[bad], equal_nan=True)
        assert np.array_equal(total[~bad, c], value[~bad, c])
        for q in np.flatnonzero(~bad):
            assert sum(Fraction(float(x)) for x in a[q]) == Fraction(float(total[q, c])), a[q]
    if kind in ("near", "cancel", "sparse", "powers"):
        assert (odd == 0).any()
    if kind in ("wide", "powers", "next to powers", "long remainders", "special"):
        assert (odd != 0).any()


@pytest.mark.parametrize("which", [0, 1])
@pytest.mark.parametrize("n,G", [(12, 1), (20, 2), (20, 3), (61, 5), (61, 16), (61, 17), (130, 33), (130, 64), (130, 70)])
def test_two_blocks_a_launch_give_the_bits_of_one(probe, n, G, which):
    """Odd and even numbers of blocks, more nodes than threads, a last block with few nodes or none."""
    N = (n + 1) ** 2
    out = []
    for two in (0, 1):
        o = np.empty((N + 2, 2))
        assert probe.probe_apply(n, G, which, two, o.ctypes.data_as(ctypes.c_void_p)) == 0
        assert o[N + 1, 1] == 0  # the ticket is back at zero
        out.append(o)
    assert np.isfinite(out[0]).all()
    assert np.array_equal(out[0].view(np.uint64), out[1].view(np.uint64))
