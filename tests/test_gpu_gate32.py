"""Gate steps: the compile-time forms against the generic launch-per-step program.

Single steps of both programs (TN_NO_FUSION: every step is a gate or a GEMM) of q = 2 and
q = 3 lattices must give the oracle's minima, on odd widths whose outer indices are no
multiples of the vector width.
"""
import numpy as np
import pytest

import instances as I
import oracle as O
import paper_2008_06888_gb300 as P

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,make,seq", [
    ("square7", lambda: I.square_lattice(7, coupling="pm1", seed=3), I.square_sweep_order(7)),
    ("square11", lambda: I.square_lattice(11, coupling="pm1", seed=4), I.square_sweep_order(11)),
    ("chimera2", lambda: I.chimera(2, coupling="pm1", seed=5), I.chimera_sweep_order(2)),
    ("potts5", lambda: I.potts_square(5, coupling="pm1", seed=6), I.square_sweep_order(5))],
    ids=lambda x: x if isinstance(x, str) else "")
def test_single_gate_steps_match_oracle(name, make, seq, monkeypatch):
    inst = make()
    ref = O.solve(inst, order=seq)
    for env in ((), ("TN_NO_FUSION",), ("TN_NO_FUSION", "TN_NO_SMALL_RUNS", "TN_NO_GATE2")):
        with monkeypatch.context() as m:
            for e in env:
                m.setenv(e, "1")
            sg = P.SpinGlass(inst, order="sweep", seq=seq)
            assert sg.energy() == ref["E"]
            assert sg.count(3)[0] == ref["count"]
