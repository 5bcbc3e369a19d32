"""Fused q = 3 chains (chain3.cu) and their traceback against one gate at a time.

Both forms add and maximise the same terms in the same order, so energies and states
must be equal bit for bit, for both value types, at the smallest tensors that take
chains (3^10), where tiles outnumber the resident blocks, alone and batched.
"""
import numpy as np
import pytest

import instances as I
import paper_2008_06888_gb300 as P

pytestmark = pytest.mark.gpu


def _orders(L):
    n = L * L
    rev = np.array(I.square_sweep_order(L))[::-1].copy()
    cols = np.arange(n).reshape(L, L).T.reshape(-1)
    return {"sweep": I.square_sweep_order(L), "reversed": rev, "columns": cols}


@pytest.mark.parametrize("L,coupling,order,B", [
    (9, "gauss", "sweep", 1), (10, "gauss", "sweep", 3), (10, "pm1", "reversed", 2),
    (11, "gauss", "columns", 2), (12, "pm1", "sweep", 1), (13, "gauss", "reversed", 2),
    (14, "gauss", "sweep", 1)])
def test_chains_equal_single_gates(L, coupling, order, B, monkeypatch):
    inst = I.potts_square(L, coupling=coupling, seed=L)
    rng = np.random.default_rng(L)
    J = rng.standard_normal((B, len(inst["J"]))).astype(np.float32)
    if coupling == "pm1":
        J = np.where(J < 0, -1, 1).astype(np.float32)
    out = []
    for fused in (True, False):
        if not fused:
            monkeypatch.setenv("TN_NO_FUSION", "1")
        sg = P.SpinGlass(inst, order="sweep", seq=_orders(L)[order])
        for _ in range(2):   # eager, then captured
            E, s = sg.config_batch(J)
        out.append((np.asarray(E), np.asarray(s), sg.energy()))
    assert np.array_equal(out[0][0], out[1][0]) and out[0][2] == out[1][2]
    e = np.asarray(inst["edges"])
    for E, s, _ in out:
        same = s[:, e[:, 0]] == s[:, e[:, 1]]
        ref = -(J.astype(np.float64) * same).sum(1)
        # a 32-bit sum of n terms: n eps of the sum of their sizes
        assert np.all(np.abs(ref - E) <= len(e) * 2.0 ** -24 * np.abs(J).sum(1))
    assert np.array_equal(out[0][1], out[1][1])
