"""Counts start the way the last ones ended: a context whose counts reach 2^59 goes to the
residue planes at once (from its second count on when the first did), and back to the
saturating run when they are small again.  Launches tell which programs ran; counts are exact either way."""
import numpy as np
import pytest

import instances as I
import oracle as O
import paper_2008_06888_gb300 as P
from paper_2008_06888_gb300 import binding as B

pytestmark = pytest.mark.gpu
L = 9
BASE = I.square_lattice(L, coupling="pm1", seed=5)
ZERO = np.zeros_like(BASE["J"])       # 2^81 ground states
SEQ = I.square_sweep_order(L)


def _sg():
    return P.SpinGlass(BASE, order="sweep", seq=SEQ)


def _launches(sg, call):
    B.tn_profile_reset(sg.ctx)
    out = call()
    return out, B.tn_profile_get(sg.ctx)["launches"]


def _alone(call_of, residues, monkeypatch):
    """Launches of the call on a fresh context that runs one program."""
    with monkeypatch.context() as m:
        if residues:
            m.setenv("TN_COUNT_RESIDUES", "1")
        sg = _sg()
        call_of(sg)()
        n = _launches(sg, call_of(sg))[1]
        sg.close()
    return n


def test_single_counts_change_their_start(monkeypatch):
    count = lambda sg: lambda: sg.count(3)[0]  # noqa: E731
    want = O.solve(BASE, order=SEQ, config=False)["count"]
    sat, res = (_alone(count, r, monkeypatch) for r in (False, True))
    assert sat != res
    sg = _sg()
    got = []
    for J in [BASE["J"]] + [ZERO] * 7 + [BASE["J"]] * 2:
        sg.set_couplings(J)
        got.append(_launches(sg, count(sg)))
    sg.close()
    assert [c for c, _ in got] == [want] + [1 << 81] * 7 + [want] * 2
    # saturated: both programs, until the running share (1/4, 7/16, ... of the last) passes
    # three quarters; then residues, the first small count still in them
    assert [n for _, n in got] == [sat] + [sat + res] * 5 + [res] * 3 + [sat]


def test_a_first_count_decides_alone(monkeypatch):
    count = lambda sg: lambda: sg.count(3)[0]  # noqa: E731
    sat, res = (_alone(count, r, monkeypatch) for r in (False, True))
    sg = _sg()
    sg.set_couplings(ZERO)
    got = [_launches(sg, count(sg)) for _ in range(3)]
    sg.close()
    assert got == [(1 << 81, n) for n in (sat + res, res, res)]


def test_one_large_count_in_three_stays_with_the_saturating_run(monkeypatch):
    count = lambda sg: lambda: sg.count(3)[0]  # noqa: E731
    sat, res = (_alone(count, r, monkeypatch) for r in (False, True))
    sg = _sg()
    got = []
    for k in range(12):
        sg.set_couplings(ZERO if k % 3 == 2 else BASE["J"])
        got.append(_launches(sg, count(sg))[1])
    sg.close()
    assert got == [sat, sat, sat + res] * 4


@pytest.mark.parametrize("zeros,route", [(0, "sat"), (1, "res"), (5, "res")])
def test_batches_of_few_elements(zeros, route, monkeypatch):
    """8 instances of 2^9 elements: one saturated one takes as long again as all."""
    J = np.stack([ZERO] * zeros + [BASE["J"]] * (8 - zeros))
    plain = np.stack([BASE["J"]] * 8)
    batch = lambda a: lambda sg: lambda: sg.count_batch(a, limbs_per=4)  # noqa: E731
    sat, res = (_alone(batch(plain), r, monkeypatch) for r in (False, True))
    want = O.solve(BASE, order=SEQ, config=False)["count"]
    sg = _sg()
    batch(J)(sg)()
    for _ in range(2):
        (E, counts, status), n = _launches(sg, batch(J)(sg))
        assert n == (sat if route == "sat" else res)
        assert list(counts) == [1 << 81] * zeros + [want] * (8 - zeros) and np.all(status == 0)
    sg.close()


def test_a_minority_of_large_instances_stays_with_the_saturating_run(monkeypatch):
    """2 of 8 instances of 2^19 elements: re-run by themselves, in every call."""
    n = 19
    base = I.square_lattice(n, coupling="pm1", seed=6)
    J = np.stack([np.zeros_like(base["J"])] * 2 + [base["J"]] * 6)
    J[:2, : len(base["J"]) // 2] = base["J"][: len(base["J"]) // 2]   # half of the bonds cut
    sg = P.SpinGlass(base, order="sweep", seq=I.square_sweep_order(n))
    out = [_launches(sg, lambda: sg.count_batch(J, limbs_per=8)) for _ in range(3)]
    monkeypatch.setenv("TN_COUNT_RESIDUES", "1")
    (E, counts, status), res = _launches(sg, lambda: sg.count_batch(J, limbs_per=8))
    sg.close()
    assert min(counts[:2]) >= 1 << 59 > max(counts[2:])
    for (Ek, ck, sk), k in out:
        assert list(ck) == list(counts) and np.array_equal(Ek, E) and np.array_equal(sk, status)
        assert k > res


def test_saturated_instances_of_many_groups_run_together(monkeypatch):
    """tn_batch_run: lattices of eight sizes, one of each size with 60% of its bonds cut.
    The re-runs of all groups are in flight together, in the groups' staging; energies,
    counts and statuses (some counts are beyond the primes' range) are those of the residue
    planes, in the first call and in the next ones."""
    insts = []
    for s in range(15, 23):
        a = [I.square_lattice(s, coupling="pm1", seed=s + k) for k in range(6)]
        J = np.array(a[0]["J"])
        J[: len(J) * 3 // 5] = 0
        insts += [dict(a[0], J=J)] + a[1:]
    sgs = [P.SpinGlass(x, order="sweep", seq=I.square_sweep_order(int(round(x["n"] ** 0.5))))
           for x in insts]

    def batch():
        st, E, counts, status = B.tn_batch_run([g.ctx for g in sgs], limbs_per=8)
        return st, list(E), list(counts), list(status)

    got = [batch() for _ in range(3)]
    monkeypatch.setenv("TN_COUNT_RESIDUES", "1")
    ref = batch()
    big = [s != B.TN_OK or c >= 1 << 59 for s, c in zip(ref[3], ref[2])]
    assert big == [k % 6 == 0 for k in range(len(insts))]
    assert ref[0] == B.TN_EOVERFLOW and ref[3].count(B.TN_EOVERFLOW) < 8
    for g in got:
        assert g == ref
    for g in sgs:
        g.close()
