"""Counts in one plane of exact 64-bit integers.

tn_count and the batched counts first run with a single 8-byte plane that
saturates at 2^64 - 1; counts that reach it run again with the residue planes
(TN_COUNT_RESIDUES starts there).  Both forms must give the oracle's integers:
all are exact, so every comparison is for equality.
"""
import numpy as np
import pytest

import instances as I
import oracle as O
import paper_2008_06888_gb300 as P
from paper_2008_06888_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2008_06888_gb300 import build
    build.build()


def _cases():
    sw = lambda L: dict(order="sweep", seq=I.square_sweep_order(L))  # noqa: E731
    # register chains with low legs at every position of the rotation, rank-raising and
    # rank-lowering ends (greedy), operands with counts above 1 (3-regular, chimera)
    yield "square14_rows", I.square_lattice(14, coupling="pm1", seed=3), sw(14)
    yield "square15_greedy", I.square_lattice(15, coupling="pm1", seed=4), \
        dict(order="greedy", seed=1, restarts=32)
    yield "square13x15_field", dict(I.square_lattice(13, 15, coupling="pm1", seed=5),
                                    h=np.random.default_rng(5).integers(-1, 2, 195)
                                    .astype(np.float32)), dict(order="greedy", seed=2)
    yield "chimera4_greedy", I.chimera(4, coupling="pm1", seed=6), dict(order="greedy", seed=2)
    yield "chimera5_cells", I.chimera(5, coupling="pm1", seed=7), \
        dict(order="sweep", seq=I.chimera_sweep_order(5))
    yield "rrg90_pm", I.random_regular3(90, coupling="pm1", seed=8), dict(order="greedy", seed=1)
    yield "potts6_pm", I.potts_square(6, coupling="pm1", seed=9), sw(6)
    yield "square12_gauss", I.square_lattice(12, coupling="gauss", seed=10), sw(12)


@pytest.mark.parametrize("case", list(_cases()), ids=lambda c: c[0])
def test_exact64_counts_match_oracle_and_residues(case, monkeypatch):
    name, inst, kw = case
    o = O.solve(inst, order=kw.get("seq"), config=False)
    sg = P.SpinGlass(inst, **kw)
    try:
        c, _, E = sg.count(3)
        monkeypatch.setenv("TN_COUNT_RESIDUES", "1")
        cr, _, Er = sg.count(3)
        assert c == cr == o["count"] and E == Er
        if name != "square12_gauss":
            assert E == o["E"]
    finally:
        sg.close()


@pytest.mark.parametrize("device", [False, True], ids=["host", "device"])
def test_saturated_instances_of_a_batch_run_with_residues(device):
    """A batch on a 14 x 14 lattice that mixes +-J couplings with zeroed ones: 2^196
    states (over three primes' range: TN_EOVERFLOW as with residues), 2^70 and 2^64
    (saturated, then exact), and counts that fit."""
    import torch
    base = I.square_lattice(14, coupling="pm1", seed=1)
    e = np.asarray(base["edges"])
    J = np.stack([I.square_lattice(14, coupling="pm1", seed=20 + k)["J"] for k in range(5)])
    J[1] = 0.0
    for k, free in ((2, 70), (4, 64)):
        # a ferromagnet on the spins from free - 1 on (2 states), the others free
        J[k] = ((e[:, 0] >= free - 1) & (e[:, 1] >= free - 1)).astype(np.float32)
    o = {k: O.solve(dict(base, J=J[k]), order=I.square_sweep_order(14), config=False)
         for k in (0, 2, 3, 4)}
    assert o[2]["count"] == 2 ** 70 and o[4]["count"] == 2 ** 64
    sg = P.SpinGlass(base, order="sweep", seq=I.square_sweep_order(14))
    try:
        Jb = torch.tensor(J, device="cuda") if device else J
        E, counts, status = sg.count_batch(Jb, limbs_per=4)
        assert status.tolist() == [0, B.TN_EOVERFLOW, 0, 0, 0]
        for k in (0, 2, 3, 4):
            assert counts[k] == o[k]["count"] and E[k] == o[k]["E"]
        assert E[1] == 0.0
    finally:
        sg.close()
    sgs = [P.SpinGlass(dict(base, J=J[k]), order="sweep", seq=I.square_sweep_order(14))
           for k in (0, 2, 3, 4)]
    try:
        st, E, counts, status = B.tn_batch_run([s.ctx for s in sgs])
        assert st == 0 and status.tolist() == [0] * 4
        assert [counts[i] for i in range(4)] == [o[k]["count"] for k in (0, 2, 3, 4)]
        assert E.tolist() == [o[k]["E"] for k in (0, 2, 3, 4)]
    finally:
        for s in sgs:
            s.close()


def test_range_of_the_primes_still_applies():
    """One prime holds counts below its 2^62 range only, although 64 bits would hold
    2^63 (J = 0 on 7 x 9 spins): refused as with residues."""
    base = I.square_lattice(7, 9, coupling="zero", seed=0)
    sg = P.SpinGlass(base, order="sweep", seq=I.square_sweep_order(7, 9))
    try:
        assert sg.count(2)[0] == 1 << 63
        with pytest.raises(B.TNError) as e:
            sg.count(1)
        assert e.value.status == B.TN_EOVERFLOW
    finally:
        sg.close()
