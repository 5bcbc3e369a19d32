"""Couplings near the largest float32 (tn_build takes every finite one): sums overflow to
infinities, and their differences to NaN.  The one-launch runs of small steps treat those
like the steps' own kernels (TN_NO_SMALL_RUNS): same energies, same states."""
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
    yield "square5", I.square_lattice(5, coupling="pm1", seed=1), dict(
        order="sweep", seq=I.square_sweep_order(5))
    yield "square9", I.square_lattice(9, coupling="pm1", seed=2), dict(order="greedy", seed=1)
    yield "rrg40", I.random_regular3(40, coupling="pm1", seed=3), dict(order="greedy", seed=1)
    yield "potts5", I.potts_square(5, coupling="pm1", seed=4), dict(order="greedy", seed=1)


@pytest.mark.parametrize("fields", [False, True])
@pytest.mark.parametrize("case", list(_cases()), ids=lambda c: c[0])
def test_overflowing_couplings(case, fields, monkeypatch):
    name, inst, kw = case
    if fields and inst["q"] == 3:
        pytest.skip("Potts instances have no fields")
    rng = np.random.default_rng(5)
    m, n, big = len(inst["J"]), inst["n"], np.float32(3.4e38)
    draw = lambda size: (np.where(rng.random(size) < 0.5, -1, 1) * big).astype(np.float32)  # noqa: E731
    J = draw((6, m))
    J[3:] *= rng.random((3, m)) < 0.3     # a few large ones among zeros: infinite both ways
    h = draw((6, n)) if fields else None
    inst = dict(inst, J=J[0], h=None if h is None else h[0])

    def results():
        sg = P.SpinGlass(inst, **kw)
        try:
            E, s = sg.config_batch(J, h)
            return [np.array(x, np.float64) for x in
                    (sg.energy(), sg.energy_batch(J, h), E, sg.config()[1])], s, sg.config()[0]
        finally:
            sg.close()

    a = results()
    monkeypatch.setenv("TN_NO_SMALL_RUNS", "1")
    b = results()
    for x, y in zip(a[0], b[0]):
        assert np.array_equal(x, y, equal_nan=True), (x, y)
    assert np.array_equal(a[1], b[1]) and np.array_equal(a[2], b[2])
    assert not np.isfinite(a[0][1]).all()
