"""Where idtx_cmi_ksg leaves its estimates, through the C ABI: host memory,
aligned device memory (stored by a kernel), and device memory that a kernel
must not store to and a copy serves, here one off the alignment of a double (the
other case, memory of another GPU, takes more than one)."""
import ctypes

import numpy as np
import pytest

from paper_1807_10459_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_result_buffers():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1807_10459_gb300 as idtx
    from paper_1807_10459_gb300 import build
    build.build()
    g = synth.gaussian_problem(300, 1, 1, 2, seed=6)
    x, y, z = (torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in (g.x, g.y, g.z))
    ctx = idtx.Context(0)
    want = idtx.cmi_ksg(x, y, z, k=4, n_surr=9, seed=3, ctx=ctx).cpu().numpy()
    s = idtx.Settings(4, 9, 3, 0.05, 0, 0)
    stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)

    def call(out):
        assert idtx.load().idtx_cmi_ksg(ctx.handle, x.data_ptr(), 1, y.data_ptr(), 1, z.data_ptr(),
                                        2, 300, 300, ctypes.byref(s), out, None, None, stream) == 0

    host = np.zeros(10)
    call(host.ctypes.data)
    assert np.array_equal(host, want)
    for offset in (0, 8, 4):
        dev = torch.zeros(96, dtype=torch.uint8, device="cuda")
        call(dev.data_ptr() + offset)
        got = dev.cpu().numpy()
        assert np.array_equal(got[offset:offset + 80].copy().view(np.float64), want)
        assert not got[:offset].any() and not got[offset + 80:].any()
