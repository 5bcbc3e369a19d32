"""Infinite couplings in the 2-to-16-state gate steps of chimera cells: a NaN first term stays
(the generic gate's rule).  Signs of the infinite energies of 48 instances as the generic
kernel, one launch per step, gives them."""
import numpy as np
import pytest

import instances as I
import paper_2008_06888_gb300 as P

pytestmark = pytest.mark.gpu

SIGNS = {2: "-----+---+-----++-+-++-+---+--+----+-+++---+---+",
         3: "+++++++++++++++++++++++++++++-++++++-+++++++++++"}


@pytest.mark.parametrize("runs", [True, False], ids=["runs", "steps"])
@pytest.mark.parametrize("L", [2, 3])
def test_chimera_cells(L, runs, monkeypatch):
    if not runs:
        monkeypatch.setenv("TN_NO_SMALL_RUNS", "1")
    sg = P.SpinGlass(I.chimera(L, coupling="gauss", seed=1), order="sweep",
                     seq=I.chimera_sweep_order(L))
    rng = np.random.default_rng(L)
    J = np.where(rng.random((48, sg.m)) < 0.2, -np.inf,
                 rng.integers(-2, 3, (48, sg.m))).astype(np.float32)
    try:
        E = sg.energy_batch(J)
    finally:
        sg.close()
    assert np.isinf(E).all()
    assert "".join("+" if x > 0 else "-" for x in E) == SIGNS[L]
