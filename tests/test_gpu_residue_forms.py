"""The forms of the residue-plane kernels against each other and the oracle.

Counts below 2^59 start with one saturating plane, so these tests ask for the residue
planes (TN_COUNT_RESIDUES): vector and scalar counting chains, 16-byte and single stores of
16-state gates, streaming, compile-time and generic gates, tiled and flat counting GEMMs,
31- and 61-bit planes.  Everything is an integer, so every comparison is for equality.
"""
import numpy as np
import pytest

import instances as I
import oracle as O
import paper_2008_06888_gb300 as P
from paper_2008_06888_gb300 import binding as B
from test_gpu_count_passes import _cases
from test_gpu_count_vec import _contiguous_16_state_gates, _low_leg_chains

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2008_06888_gb300 import build
    build.build()


@pytest.fixture(autouse=True)
def residues(monkeypatch):
    monkeypatch.setenv("TN_COUNT_RESIDUES", "1")


def _count(make, monkeypatch, **env):
    """(count, E) of a fresh context with the switches of `env` set, twice (eager, graph)."""
    with monkeypatch.context() as m:
        for k, v in env.items():
            m.setenv(k, v)
        sg = make()
        try:
            a, b = sg.count(3), sg.count(3)
            assert a == b
            return a[0], a[2]
        finally:
            sg.close()


@pytest.mark.parametrize("L,seed", [(11, 4), (12, 8)])
def test_vector_and_scalar_chains(L, seed, monkeypatch):
    assert _low_leg_chains(L, seed) > 0
    inst, seq = I.square_lattice(L, coupling="pm1", seed=seed), I.square_sweep_order(L)
    o = O.solve(inst, order=seq, config=False)
    make = lambda: P.SpinGlass(inst, order="sweep", seq=seq)  # noqa: E731
    vec = _count(make, monkeypatch)
    assert vec == _count(make, monkeypatch, TN_RCC_NO_VEC="1") == (o["count"], o["E"])


def test_vector_and_scalar_chains_in_a_mixed_batch(monkeypatch):
    insts = I.mixed_square_batch(24, Lmin=8, Lmax=14, seed=77)

    def run():
        sgs = [P.SpinGlass(x, order="sweep", seq=I.square_sweep_order(int(np.sqrt(x["n"]))))
               for x in insts]
        try:
            st, E, counts, status = B.tn_batch_run([s.ctx for s in sgs])
            return st, list(E), list(counts), list(status)
        finally:
            for s in sgs:
                s.close()

    a = run()
    monkeypatch.setenv("TN_RCC_NO_VEC", "1")
    assert a[0] == 0 and a == run()
    monkeypatch.delenv("TN_COUNT_RESIDUES")
    assert a == run()


@pytest.mark.parametrize("L,seed", [(4, 2), (5, 7)])
def test_forms_of_cell_gates(L, seed, monkeypatch):
    assert _contiguous_16_state_gates(L, seed) > 0
    inst, seq = I.chimera(L, coupling="pm1", seed=seed), I.chimera_sweep_order(L)
    o = O.solve(inst, order=seq, config=False)
    make = lambda: P.SpinGlass(inst, order="sweep", seq=seq)  # noqa: E731
    for env in ({}, {"TN_GATE_TC_NO_VEC": "1"}, {"TN_NO_GATE_TC": "1"},
                {"TN_NO_GATE_TC": "1", "TN_NO_GATE2": "1"}):
        assert _count(make, monkeypatch, **env) == (o["count"], o["E"]), env


@pytest.mark.parametrize("kind", ["sat", "square_pm", "potts"])
def test_streaming_and_generic_gates(kind, monkeypatch):
    if kind == "sat":
        sat = I.max2sat_regular3(120, seed=6)
        make = lambda: P.Max2SAT(sat, order="greedy", seed=2, restarts=64)  # noqa: E731
    elif kind == "square_pm":
        inst = I.square_lattice(14, coupling="pm1", seed=3)
        make = lambda: P.SpinGlass(inst, order="greedy", seed=2, restarts=64)  # noqa: E731
    else:
        inst = I.potts_square(8, coupling="pm1", seed=3)
        make = lambda: P.SpinGlass(inst, order="greedy", seed=2, restarts=64)  # noqa: E731
    ref = _count(make, monkeypatch)
    for env in ({"TN_NO_GATE2": "1"}, {"TN_NO_GATE2": "1", "TN_NO_GATE_TC": "1"}):
        assert _count(make, monkeypatch, **env) == ref, env


@pytest.mark.parametrize("case", list(_cases())[:4], ids=lambda c: c[0])
def test_31_and_61_bit_planes(case, monkeypatch):
    name, inst, kw = case
    o = O.solve(inst, order=kw.get("seq"), config=False)
    make = lambda: P.SpinGlass(inst, **kw)  # noqa: E731
    c, E = _count(make, monkeypatch)
    assert c == o["count"]
    assert (c, E) == _count(make, monkeypatch, TN_COUNT_61="1")


def test_tiled_and_flat_gemms(monkeypatch):
    inst = I.chimera(4, coupling="pm1", seed=5)
    o = O.solve(inst, order=I.chimera_sweep_order(4), config=False)

    def make():
        sg = P.SpinGlass(inst, order="greedy", seed=2, restarts=16)
        assert B.tn_plan_launches(sg.ctx, "count")["gemm"] > 0
        return sg

    tiled = _count(make, monkeypatch)
    assert tiled == _count(make, monkeypatch, TN_GEMM_COUNT_FLAT="1") == (o["count"], o["E"])
