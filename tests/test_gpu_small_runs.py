"""Small contraction steps grouped into runs (one launch, one block per instance).

The runs keep every step's operands and order of terms, so energies, counts and
ground states must equal those of the launch-per-step program (TN_NO_SMALL_RUNS)
bit for bit, for both value types, Ising and Potts digits, transposes and GEMM
steps, alone and batched.
"""
import numpy as np
import pytest

import instances as I
import paper_2008_06888_gb300 as P

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2008_06888_gb300 import build
    build.build()


def _cases():
    for L in (1, 2, 5, 13):   # one spin; all steps small; the state outgrows the runs
        yield f"square{L}_pm", I.square_lattice(L, coupling="pm1", seed=L), \
            dict(order="sweep", seq=I.square_sweep_order(L))
    yield "square14_gauss_h", I.square_lattice(14, coupling="gauss", field_sigma=0.1, seed=2), \
        dict(order="greedy", seed=1)
    yield "chimera3_pm", I.chimera(3, coupling="pm1", seed=3), dict(order="greedy", seed=2)
    yield "chimera4_pm", I.chimera(4, coupling="pm1", seed=3), \
        dict(order="sweep", seq=I.chimera_sweep_order(4))
    yield "rrg120_gauss", I.random_regular3(120, coupling="gauss", seed=4), \
        dict(order="greedy", seed=1, restarts=32)
    yield "potts7_gauss", I.potts_square(7, coupling="gauss", seed=5), dict(order="greedy", seed=1)


@pytest.mark.parametrize("case", list(_cases()), ids=lambda c: c[0])
def test_runs_equal_single_steps(case, monkeypatch):
    name, inst, kw = case
    rng = np.random.default_rng(1)
    scale = rng.integers(1, 4, (3, len(inst["J"]))).astype(np.float32)
    Jb = scale * inst["J"]
    hb = None if inst["h"] is None else np.stack([inst["h"]] * 3)

    def results():
        sg = P.SpinGlass(inst, **kw)
        try:
            s, E = sg.config()
            c, _, Ec = sg.count(3)
            Eb, cb, st = sg.count_batch(Jb, hb, limbs_per=4)
            Es, sb = sg.config_batch(Jb, hb)
            return ([sg.energy(), E, c, Ec, s.tolist(), Eb.tolist(), cb, st.tolist(), Es.tolist(),
                     sb.tolist()])
        finally:
            sg.close()

    a = results()
    monkeypatch.setenv("TN_NO_SMALL_RUNS", "1")
    assert a == results()
