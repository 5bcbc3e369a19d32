"""Samples from the tables of one sweep equal those of the prefix-by-prefix counts.

Both draw the same random integers below the same exact counts, so the samples must be
equal element by element: across the widths where the sweep changes from one block to a
launch per step (2^13 states), records that do not fit the staged chunks, any order,
fields, isolated spins, and counts that saturate.
"""
import os
import shutil
import subprocess

import numpy as np
import pytest

import instances as I
import paper_2008_06888_gb300 as P

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2008_06888_gb300", "csrc")


def test_frontier_tables_with_brute_force_counts(tmp_path):
    """tests/host/frontier_check.cpp: plans of random graphs and orders."""
    if shutil.which("g++") is None:
        pytest.skip("g++ missing")
    exe = str(tmp_path / "frontier_check")
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", CSRC,
                    os.path.join(ROOT, "tests", "host", "frontier_check.cpp"),
                    os.path.join(CSRC, "sampler.cpp"), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=240)
    assert r.returncode == 0, r.stdout + r.stderr


def _complete(n, seed):
    e = np.array([(i, j) for i in range(n) for j in range(i)], np.int32)
    rng = np.random.default_rng(seed)
    return dict(n=n, q=2, edges=e, J=(rng.integers(0, 2, len(e)) * 2 - 1).astype(np.float32), h=None)


CASES = {
    "square5_h": lambda: (I.square_lattice(5, coupling="pm1", seed=1), True, 33, None),
    "square13": lambda: (I.square_lattice(13, coupling="pm1", seed=2), False, 2, None),
    "square14": lambda: (I.square_lattice(14, coupling="pm1", seed=3), False, 2, None),
    "reversed7": lambda: (I.square_lattice(7, coupling="pm1", seed=4), False, 3, "rev"),
    "shuffled6": lambda: (I.square_lattice(6, coupling="pm1", seed=5), True, 3, "rand"),
    "complete20": lambda: (_complete(20, 6), False, 1, None),   # 190 neighbour entries
    "free": lambda: (dict(n=61, q=2, edges=np.zeros((0, 2), np.int32),
                          J=np.zeros(0, np.float32), h=None), False, 2, None),   # 2^61 states
}


@pytest.mark.gpu
@pytest.mark.parametrize("name", list(CASES))
def test_samples_equal_prefix_counts(name, monkeypatch):
    inst, fields, S, order = CASES[name]()
    n = inst["n"]
    if fields:
        inst = dict(inst, h=np.random.default_rng(9).integers(-1, 2, n).astype(np.float32))
    order = {None: None, "rev": np.arange(n)[::-1],
             "rand": np.random.default_rng(8).permutation(n)}[order]
    sg = P.SpinGlass(inst, order="greedy", seed=1, restarts=16)
    got = sg.sample(S, seed=11, order=order)
    again = sg.sample(S, seed=11, order=order)
    E, _ = sg.config_batch(np.asarray(inst["J"], np.float32)[None],
                           None if inst["h"] is None else np.asarray(inst["h"])[None]) \
        if len(inst["J"]) else (None, None)
    monkeypatch.setenv("TN_COUNT_RESIDUES", "1")
    want = sg.sample(S, seed=11, order=order)
    assert np.array_equal(got, want) and np.array_equal(again, want)
    if E is not None:
        e = np.asarray(inst["edges"])
        h = 0.0 if inst["h"] is None else got @ np.asarray(inst["h"], np.float64)
        assert np.all(-(got[:, e[:, 0]] * got[:, e[:, 1]]) @ np.asarray(inst["J"], np.float64) - h
                      == E[0])
