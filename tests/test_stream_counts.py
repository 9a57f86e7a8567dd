"""The stream schedule's load counts, which decide whether a handle may take it, against the lists that a
handle builds when it walks its trees."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_2605_19928_gb300 import capi, synth

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2605_19928_gb300", "csrc")


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not found")
    out = str(tmp_path_factory.mktemp("count_probe") / "libcountprobe.so")
    subprocess.run([gxx, "-O1", "-std=c++17", "-fPIC", "-shared", "-I", os.path.join(ROOT, "include"), "-I", CSRC,
                    os.path.join(ROOT, "tests", "count_probe.cpp"), os.path.join(CSRC, "tree.cpp"), "-o", out],
                   check=True, capture_output=True)
    return C.CDLL(out)


def _leaf_turn():
    g = synth.turn_subgame(n_hands=9, seed=3, range_seed=4, bet_sizes=(1.0, synth.ALL_IN), max_raises=2)
    g.depth_limit = 1
    return g


@pytest.mark.parametrize("make", [
    synth.kuhn, synth.leduc, lambda: synth.river_subgame(n_hands=5, max_raises=0),
    lambda: synth.river_subgame(n_hands=40, bet_sizes=(0.33, 0.5, 0.75, 1.0, 2.0, synth.ALL_IN), stack=900.0),
    lambda: synth.turn_subgame(n_hands=12, bet_sizes=(synth.ALL_IN,), max_raises=1), _leaf_turn])
@pytest.mark.parametrize("pred", [0, 1])
def test_counts_are_those_of_the_lists(probe, make, pred):
    spec, keep = capi.make_spec(make())
    out = np.zeros(10, np.int32)
    assert probe.probe_counts(C.byref(spec), pred, out.ctypes.data_as(C.c_void_p)) == 0
    assert out[:5].tolist() == out[5:].tolist() and out[4] > 0
