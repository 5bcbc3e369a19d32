"""Products of gate contractions in one step (gate_sum.cu) against separate steps.

Sums, maxima and products are those of the separate steps in their order, so energies
and counts must be equal, for both value types, rows of K_{4,4} cells of several widths
(products of two, of four, and what is left over), alone and batched, and with counts
that saturate.
"""
import numpy as np
import pytest

import instances as I
import paper_2008_06888_gb300 as P

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,coupling,order", [
    (2, "pm1", "sweep"), (3, "pm1", "sweep"), (3, "gauss", "sweep"), (4, "pm1", "sweep"),
    (4, "gauss", "sweep"), (4, "pm1", "greedy"), (5, "pm1", "sweep")])
def test_products_equal_separate_steps(L, coupling, order, monkeypatch):
    inst = I.chimera(L, coupling=coupling, seed=L)
    kw = dict(order="sweep", seq=I.chimera_sweep_order(L)) if order == "sweep" else \
        dict(order="greedy", seed=2, restarts=8)
    B = 3 if L < 5 else 1
    rng = np.random.default_rng(L)
    J = rng.standard_normal((B, len(inst["J"]))).astype(np.float32)
    if coupling == "pm1":
        J = np.where(J < 0, -1, 1).astype(np.float32)
    out = []
    for fused in (True, False):
        if not fused:
            monkeypatch.setenv("TN_NO_GATE_SUM", "1")
        sg = P.SpinGlass(inst, **kw)
        r = []
        for _ in range(2):   # eager, then captured
            r.append((sg.energy(), sg.count(3), list(sg.energy_batch(J)),
                      [np.asarray(x).tolist() for x in sg.count_batch(J, None, 3, limbs_per=4)]))
        assert r[0] == r[1]
        out.append(r[0])
    assert out[0] == out[1]


def test_products_with_saturating_counts():
    """No couplings: every state is a ground state, 2^72 of them on 3 x 3 cells."""
    inst = I.chimera(3, coupling="pm1", seed=1)
    inst = dict(inst, J=np.zeros(len(inst["J"]), np.float32))
    sg = P.SpinGlass(inst, order="sweep", seq=I.chimera_sweep_order(3))
    assert sg.count(3)[0] == 2 ** 72
