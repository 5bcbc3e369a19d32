"""The count arena that tn_plan_info reports holds any count: the residue planes' one, which
a count of 2^59 and more needs, not only the saturating run's (host only)."""
import pytest

import instances as I
import paper_2008_06888_gb300 as P


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2008_06888_gb300 import build
    build.build()


CASES = [("square", I.square_lattice(14, coupling="pm1", seed=1), I.square_sweep_order(14)),
         ("square_gauss", I.square_lattice(12, coupling="gauss", seed=1), I.square_sweep_order(12)),
         ("chimera", I.chimera(4, coupling="pm1", seed=1), I.chimera_sweep_order(4)),
         ("potts", I.potts_square(6, coupling="pm1", seed=1), I.square_sweep_order(6)),
         ("small", I.square_lattice(3, coupling="pm1", seed=1), I.square_sweep_order(3))]


@pytest.mark.parametrize("name,inst,seq", CASES, ids=[c[0] for c in CASES])
def test_count_arena_holds_the_residue_planes(name, inst, seq, monkeypatch):
    sg = P.SpinGlass(inst, order="sweep", seq=seq)
    try:
        got = sg.plan_info()["arena_count"]
        monkeypatch.setenv("TN_COUNT_RESIDUES", "1")
        assert got >= sg.plan_info()["arena_count"]
    finally:
        sg.close()
