"""Tensor memory shared by CTAs of different launches (csrc/tmem_share.cuh), checked on the host: whatever CTAs fit an
SM's shared memory, their tensor-memory columns fit too, so that no allocation waits for columns held by a CTA that
itself waits for cluster or grid peers (two policy calls on two streams)."""
import ctypes
import itertools
import os
import subprocess

import pytest

from paper_2606_31315_gb300 import _build

SM = 228 * 1024  # shared memory of an sm_103 SM
BLOCK = 1024     # the system's share per CTA


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    d = tmp_path_factory.mktemp("tmem_share")
    src, lib = d / "rule.cc", d / "rule.so"
    src.write_text('#include "tmem_share.cuh"\n'
                   'extern "C" int columns(int n) { return bp::tmem_columns(n); }\n'
                   'extern "C" int share(int c, int sm) { return bp::tmem_smem_share(c, sm); }\n')
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", f"-I{_build.CSRC}", str(src), "-o", str(lib)], check=True)
    return ctypes.CDLL(os.fspath(lib))


def _most_columns(kinds):
    """Most tensor-memory columns that CTAs of these (columns, shared memory) kinds can ask for on one SM."""
    best = [0] * (SM + 1)
    for cols, smem in kinds:
        for room in range(smem, SM + 1):
            best[room] = max(best[room], best[room - smem] + cols)
    return best[SM]


def test_any_mix_of_launches_fits(rule):
    kinds = [(c, rule.share(c, SM)) for c in (32, 64, 128, 256, 512)]
    assert _most_columns(kinds) == 512


@pytest.mark.parametrize("a, b", list(itertools.combinations_with_replacement((16, 32, 48, 64), 2)))
def test_pairs_of_policy_calls_fit(rule, a, b):
    """One-shot calls take four accumulators of npad columns, streamed ones one."""
    cols = [rule.columns(n * k) for n in (a, b) for k in (1, 4)]
    assert all(c >= n * k for c, (n, k) in zip(cols, ((n, k) for n in (a, b) for k in (1, 4))))
    assert _most_columns([(c, rule.share(c, SM)) for c in cols]) <= 512


def test_a_launch_of_one_kind_keeps_its_residency(rule):
    """The share leaves 512 / columns CTAs of a launch to an SM, and fits a CTA's limit of 227 KB."""
    for c in (32, 64, 128, 256, 512):
        assert rule.columns(c) == c and rule.columns(c - 1) == c
        assert (512 // c) * rule.share(c, SM) <= SM
        assert rule.share(c, SM) - BLOCK <= 227 * 1024
