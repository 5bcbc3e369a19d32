"""Which steps the one-launch runs take: up to 1024 outputs and 4096 products (host only,
from the launches of the lowered energy program)."""
import pytest

import instances as I
import paper_2008_06888_gb300 as P
from paper_2008_06888_gb300 import binding as B


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2008_06888_gb300 import build
    build.build()


def _launches(inst, **kw):
    sg = P.SpinGlass(inst, **kw)
    try:
        n = B.tn_plan_launches(sg.ctx, "energy")
        return sum(n.values())
    finally:
        sg.close()


@pytest.mark.parametrize("L", [9, 11])
def test_steps_of_2048_outputs_keep_their_own_launches(L):
    """Row by row, an L x L lattice has one contraction of 2^L outputs and 2^(L + 1)
    products per spin of the bulk: inside a run at L = 9, a launch each at L = 11 (where
    the one block of a run would take them two outputs per thread and more, in turn)."""
    n = _launches(I.square_lattice(L, coupling="gauss", field_sigma=0.1, seed=1), order="sweep",
                  seq=I.square_sweep_order(L))
    if L == 9:
        assert n <= 4
    else:
        assert n >= (L - 2) * L


def test_few_outputs_with_many_products_stay_in_a_run():
    """A greedy order of a 10 x 10 lattice ends in contractions of 256 to 1024 outputs and
    2048 to 4096 products."""
    assert _launches(I.square_lattice(10, coupling="pm1", seed=11), order="greedy", seed=1,
                     restarts=32) <= 10
