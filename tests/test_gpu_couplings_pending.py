"""Host couplings that are replaced, or whose context changes its stream, while their
upload is still queued: tn_forward without an energy returns without a wait."""
import ctypes as C

import numpy as np
import pytest
import torch

import instances as I
import paper_2008_06888_gb300 as P
from paper_2008_06888_gb300 import binding as B

pytestmark = pytest.mark.gpu


def _queue_work(stream):
    """A few tens of milliseconds of work on a stream, and an event behind it."""
    with torch.cuda.stream(stream):
        x = torch.zeros((8192, 8192), dtype=torch.bfloat16, device="cuda")
        torch.cuda.synchronize()
        for _ in range(40):
            y = x @ x
        ev = torch.cuda.Event()
        ev.record(stream)
    return ev, (x, y)


def _couplings(inst, rng, fields):
    J = np.where(rng.integers(0, 2, len(inst["J"])) == 0, -1, 1).astype(np.float32)
    return J, rng.integers(-1, 2, inst["n"]).astype(np.float32) if fields else None


def _setup(fields):
    inst = I.square_lattice(6, coupling="pm1", seed=1)
    rng = np.random.default_rng(11)
    if fields:
        inst = dict(inst, h=rng.integers(-1, 2, inst["n"]).astype(np.float32))
    sets = [_couplings(inst, rng, fields) for _ in range(2)]
    seq = I.square_sweep_order(6)
    sg = P.SpinGlass(inst, order="sweep", seq=seq)
    want = []
    for J, h in sets:
        ref = P.SpinGlass(dict(inst, J=J, h=h), order="sweep", seq=seq)
        want.append((ref.config(), ref.energy(), ref.count(3)))
        ref.close()
    s = torch.cuda.Stream()
    sg.set_stream(s.cuda_stream)
    sg.config()
    sg.energy()
    return sg, s, sets, want


def _forward(sg):
    assert B.lib().tn_forward(sg.ctx, C.POINTER(C.c_double)()) == B.TN_OK


@pytest.mark.parametrize("fields", [False, True])
def test_couplings_replaced_behind_a_queued_upload(fields):
    sg, s, sets, want = _setup(fields)
    sg.set_couplings(*sets[0])
    ev, keep = _queue_work(s)
    _forward(sg)                 # queues the upload of the first set
    sg.set_couplings(*sets[1])   # rewrites the arrays that it reads
    assert ev.query()            # so it has to wait for the upload, and for the work before it
    sigma = B.tn_backward(sg.ctx, sg.n)
    assert np.array_equal(sigma, want[0][0][0])
    assert sg.energy() == want[1][1] and sg.count(3) == want[1][2]
    sg.close()


@pytest.mark.parametrize("fields", [False, True])
def test_stream_changed_behind_a_queued_upload(fields):
    sg, s, sets, want = _setup(fields)
    t = torch.cuda.Stream()
    sg.set_couplings(*sets[0])
    ev, keep = _queue_work(s)
    _forward(sg)
    sg.set_stream(t.cuda_stream)
    assert ev.query()            # the uploaded values are there before the new stream reads them
    assert sg.energy() == want[0][1] and sg.count(3) == want[0][2]
    sg.close()


def test_context_freed_behind_a_queued_upload():
    sg, s, sets, want = _setup(True)
    sg.set_couplings(*sets[0])
    ev, keep = _queue_work(s)
    _forward(sg)
    sg.close()
    assert ev.query()
    torch.cuda.synchronize()
