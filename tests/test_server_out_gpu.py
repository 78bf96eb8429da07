"""GPU: results of the server written to host memory at any address: whole
lines, a line's middle, one value off and an address no kernel can store to;
nothing beside the result is written."""
import numpy as np
import pytest

from synth import gaussian_pulse, jittered_delaunay_mesh

pytestmark = pytest.mark.gpu
PAD = 256  # bytes around the result


@pytest.mark.parametrize("n,N", [(1, 1), (3, 4), (20, 3), (40, 7)])  # K Np = 6 ... 115,200
def test_results_at_any_address(n, N):
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1304_5546_gb300 import build as B
    B.build()
    import paper_1304_5546_gb300 as P
    s = P.Solver(*jittered_delaunay_mesh(n, seed=2), N=N, precision="fp32")
    q0 = np.stack(gaussian_pulse(*s.nodes(), 0.5, 0.5, 0.2)).astype(np.float32)
    nbytes = 3 * s.K * s.Np * 4
    cap = [0] * 7
    cap[N - 1] = 4 * ((s.K + 3) // 4 * 4)
    srv = P.Server(cap)
    outs = []
    for off in (0, 4, 60, 1):
        buf = np.full(nbytes + 2 * PAD, 0xA5, np.uint8)
        at = PAD + (-(buf.ctypes.data + PAD)) % 128 + off - 128
        out = np.frombuffer(buf.data, np.float32, 3 * s.K * s.Np, at).reshape(3, s.K, s.Np)
        outs.append((buf, at, out, srv.submit(s, 2.5 * s.cfl_dt(), q0=q0, out=out)))
    for *_, rid in outs:
        srv.wait(rid)
    want = np.array(outs[0][2])
    assert np.isfinite(want).all() and np.abs(want).max() > 0
    for buf, at, out, _ in outs:
        np.testing.assert_array_equal(np.array(out), want)
        assert (buf[:at] == 0xA5).all() and (buf[at + nbytes:] == 0xA5).all()
    srv.close()
