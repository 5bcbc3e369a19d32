"""Host couplings are uploaded without waiting: every change reaches the next call,
also when the stream changes between the upload and the call, with and without fields."""
import numpy as np
import pytest
import torch

import instances as I
import paper_2008_06888_gb300 as P
from paper_2008_06888_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fields", [False, True])
def test_changes_reach_the_next_call(fields):
    inst = I.square_lattice(6, coupling="pm1", seed=1)
    n, rng = inst["n"], np.random.default_rng(3)
    if fields:
        inst = dict(inst, h=rng.integers(-1, 2, n).astype(np.float32))
    seq = I.square_sweep_order(6)
    sg = P.SpinGlass(inst, order="sweep", seq=seq)
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    for k in range(6):
        J = np.where(rng.integers(0, 2, len(inst["J"])) == 0, -1, 1).astype(np.float32)
        h = rng.integers(-1, 2, n).astype(np.float32) if fields else None
        ref = P.SpinGlass(dict(inst, J=J, h=h), order="sweep", seq=seq)
        sg.set_couplings(J, h)
        if k % 2:
            # an upload on one stream (the traceback has not run: refused after it) ...
            sg.set_stream(streams[0].cuda_stream)
            with pytest.raises(Exception):
                B.tn_backward(sg.ctx, None)
            B.tn_forward(sg.ctx)
        # ... and its use on another
        sg.set_stream(streams[k % 2].cuda_stream)
        assert sg.energy() == ref.energy()
        assert sg.count(3) == ref.count(3)


def test_stream_change_inside_a_capture():
    """tn_set_stream after an upload leaves a capture of the caller's work alone."""
    inst = I.square_lattice(6, coupling="pm1", seed=2)
    sg = P.SpinGlass(inst, order="sweep", seq=I.square_sweep_order(6))
    E = sg.energy()
    x = torch.zeros(8, device="cuda")
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, capture_error_mode="global"):
        sg.set_stream(torch.cuda.current_stream().cuda_stream)
        x += 1
    g.replay()
    torch.cuda.synchronize()
    sg.set_stream(0)
    assert float(x.sum()) == 8.0 and sg.energy() == E
