"""The traceback of folded q = 2 plans: chain records of 4, 5 and 6 register legs
(TN_REG_BITS), rank-changing chains, plain records and records wide enough for a grid
search.  The instances have unique ground states, so sigma must be the oracle's."""
import numpy as np
import pytest

import instances as I
import oracle as O
import paper_2008_06888_gb300 as P

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2008_06888_gb300 import build
    build.build()


def _cases():
    yield "square15_rows", I.square_lattice(15, coupling="gauss", field_sigma=0.3, seed=1), \
        dict(order="sweep", seq=I.square_sweep_order(15))
    yield "square14x16_greedy", I.square_lattice(14, 16, coupling="gauss", field_sigma=0.3,
                                                 seed=2), dict(order="greedy", seed=3)
    c = I.chimera(4, coupling="gauss", seed=3)
    # the root step contracts 2^16 states; integral fields and couplings too
    yield "chimera4_cells", dict(c, h=np.random.default_rng(3).standard_normal(128)
                                 .astype(np.float32)), \
        dict(order="sweep", seq=I.chimera_sweep_order(4))
    ints = np.random.default_rng(4)
    s = I.square_lattice(14, coupling="pm1", seed=4)
    yield "square14_ints", dict(s, J=ints.integers(-5000, 5000, len(s["J"])).astype(np.float32),
                                h=ints.integers(-500, 500, 196).astype(np.float32)), \
        dict(order="greedy", seed=1)


@pytest.mark.parametrize("bits", ["4", "5", "6"])
@pytest.mark.parametrize("case", list(_cases()), ids=lambda c: c[0])
def test_walk_finds_the_oracles_state(case, bits, monkeypatch):
    name, inst, kw = case
    monkeypatch.setenv("TN_REG_BITS", bits)
    o = O.solve(inst, order=kw.get("seq"), count=False)
    sg = P.SpinGlass(inst, **kw)
    try:
        s, E = sg.config()
        assert np.array_equal(P.SpinGlass.state_indices(s, 2), o["state"].astype(np.int8))
        # values are float32 sums: the oracle's energy within its stated tolerance
        assert abs(E - o["E"]) <= 1e-5 * max(1.0, abs(o["E"]))
        Jb = np.stack([inst["J"], -inst["J"]])
        _, sb = sg.config_batch(Jb, np.stack([inst["h"]] * 2))
        assert np.array_equal(sb[0], s)
    finally:
        sg.close()
