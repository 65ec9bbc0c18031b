"""Steps of small grids beside channels: a receive that polls on another stream for a message that stands behind the step must not keep
the step out, so no resident launch is issued while a channel is open on the device."""
import numpy as np
import pytest
import torch

import jacobi_inputs as J
import oracle

pytestmark = pytest.mark.gpu

GRID, SPLIT = (128, 128, 128), ("shape", (32, 32, 32))
INIT = dict(bc="uniform", bc_seed=3, interior="zero")


@pytest.mark.parametrize("own", [True, False])
@pytest.mark.parametrize("zero_copy", [True, False])
@pytest.mark.parametrize("path", ["graph", "persistent"])
def test_receive_polls_while_the_step_is_queued(path, zero_copy, own):
    """Stream a: a step, then the send; stream b: its receive.  Zero-copy it is issued first, else after the send, which the step keeps
    back.  `own`: the channel belongs to the stepping handle, else to another one.  The receive is one CTA: one that polls on every SM
    (2.4 MB or more) can keep any step out, since an SM divides its memory anew only when it is empty."""
    import paper_2102_12416_gb300 as jg
    u = J.initial_grid(*GRID, dtype=np.float32, **INIT)
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    n = 16 << 10
    src = torch.arange(n, device="cuda", dtype=torch.int64).to(torch.uint8)
    dst = torch.zeros_like(src)
    torch.cuda.synchronize()
    with jg.Jacobi3D(GRID, SPLIT, "f32", INIT, path=path, stream=a) as s, jg.Jacobi3D((8, 8, 8), ("count", (2, 1, 1)), "f32") as o:
        ch = jg.channel_open(s.h if own else o.h, 1, 0, 1, n)
        # all kernels once, in an order without a wait: loading one synchronises with those that run
        s.step(40)
        for d in (None, dst.data_ptr()):
            jg.channel_send(ch, 0, src.data_ptr(), n, a)
            jg.channel_recv(ch, 1, d, n, a)
        jg.channel_sync(ch, a)
        dst.zero_()
        torch.cuda.synchronize()
        if zero_copy:
            jg.channel_recv(ch, 1, None, n, b)
        s.step(40)
        jg.channel_send(ch, 0, src.data_ptr(), n, a)
        if not zero_copy:
            jg.channel_recv(ch, 1, dst.data_ptr(), n, b)
        jg.channel_sync(ch, a)
        jg.channel_sync(ch, b)  # neither waited in vain
        assert s.info.resident_launches == 0
        if not zero_copy:
            assert torch.equal(dst, src)
        assert np.array_equal(s.copy_out(), J.interior_of(oracle.jacobi(u, 80)))
        jg.channel_close(ch)
        s.step(40)
        assert s.info.resident_launches == 1
        assert np.array_equal(s.copy_out(), J.interior_of(oracle.jacobi(u, 120)))


def test_gate_counts_open_channels():
    import paper_2102_12416_gb300 as jg

    def runs(s):
        before = s.info.resident_launches
        s.step(40)
        return s.info.resident_launches > before

    with jg.Jacobi3D((32, 32, 32), ("count", (2, 2, 2)), "f64", path="graph") as s:
        assert runs(s)
        o = jg.Jacobi3D((8, 8, 8), ("count", (2, 1, 1)), "f32")
        c1, c2 = jg.channel_open(o.h, 1, 0, 1, 64), jg.channel_open(o.h, 2, 0, 1, 64)
        with pytest.raises(jg.JacobiError):
            jg.channel_open(o.h, 2, 0, 1, 64)  # refused: not counted
        assert not runs(s)
        jg.channel_close(c1)
        assert not runs(s)
        o.close()  # closes c2
        assert c2 and runs(s)
