"""The rules that choose how a level or a launch runs (csrc/hz_rules.h), on the CPU."""
import ctypes
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1312_2880_gb300", "csrc")
SMS = 152


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("rules") / "rules.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I" + CSRC, os.path.join(HERE, "rules_probe.cpp"),
                    "-o", so], check=True)
    return ctypes.CDLL(so)


def test_a_tuned_fp64_pass_is_not_reused_for_another_operator_kind(rules):
    d = ctypes.c_double
    kinds = [(0.0, 0.0), (0.5, 0.0), (0.5, 0.5)]  # L / L, M / L, M / M
    for q, a in enumerate(kinds):
        for r, b in enumerate(kinds):
            key = lambda up, fp32: rules.same_tuning(2048, 1, up, 0, fp32, d(a[0]), d(a[1]), d(b[0]), d(b[1]))
            assert key(0, 0) == (q == r)  # the pass down relaxes and forms the residual
            assert key(1, 0) == ((a[0] == 0) == (b[0] == 0))  # the pass up only relaxes
            assert key(0, 1) == key(1, 1) == 1  # FP32: one code for every operator
    assert rules.same_tuning(2048, 1, 0, 0, 0, d(0.5), d(0.5), d(0.3), d(0.3))
    assert not rules.same_shape(2048, 1024, 1, 1) and not rules.same_shape(2048, 2048, 1, 2)


def test_large_batches_of_passes_take_the_largest_tiles(rules):
    """From four waves of the 62-node tiles on: there the halo decides (n_l = 128 with 64 and 152 right-hand sides)."""
    for n, batch in ((128, 64), (128, 152), (136, 64), (144, 152), (224, 64)):
        assert rules.pass_cfg(n, 4, batch, SMS) == 2, (n, batch)
    for n, nu, batch, want in ((128, 4, 1, 0), (128, 2, 1, 1), (192, 4, 1, 1), (256, 4, 1, 1), (128, 4, 16, 2), (96, 4, 8, 1)):
        assert rules.pass_cfg(n, nu, batch, SMS) == want, (n, nu, batch)


def test_two_sweep_tiles_where_whole_passes_lose(rules):
    for n in (448, 512, 543):  # the 37-node tiles take a second wave, two 32-node tiles come on an SM
        assert rules.pass_cfg(n, 4, 1, SMS) == 3 and rules.pass_cfg(n, 8, 1, SMS) == 3, n
        assert rules.pass_cfg(n, 4, 8, SMS) == 2, n
    for n in (416, 443, 544, 576, 704, 743):
        assert rules.pass_cfg(n, 4, 1, SMS) in (1, 2), n
    for n in (744, 1024, 2048, 16384):
        assert rules.pass_cfg(n, 4, 1, SMS) == rules.pass_cfg(n, 4, 2, SMS) == 4, n
    for n in (448, 512, 1024, 2048):  # an odd number of two-sweep launches would not end in its own array
        assert rules.pass_cfg(n, 2, 1, SMS) in (1, 2) and rules.pass_cfg(n, 6, 1, SMS) in (1, 2), n


def test_the_operator_rule_counts_all_right_hand_sides(rules):
    for n, batch, want in ((512, 1, 1), (511, 1, 0), (128, 1, 0), (128, 15, 0), (128, 16, 1), (64, 64, 1), (16384, 1, 1)):
        assert rules.fills_gpu(ctypes.c_longlong((n + 1) ** 2), batch) == want, (n, batch)


def test_batches_of_ragged_levels_take_clusters(rules):
    """n_l = 124 .. 161, three 62-node tiles each way, from 17 right-hand sides (two waves of them) on."""
    for n, batch, want in ((136, 17, 1), (136, 16, 0), (136, 1, 0), (124, 24, 1), (161, 24, 1), (123, 64, 0), (162, 64, 0),
                           (256, 64, 0)):
        assert rules.ragged_batch(n, batch, SMS) == want, (n, batch)
