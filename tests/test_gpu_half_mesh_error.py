"""The split two-band k-sum over half of the fine mesh is as accurate as the sum over all of it (the kernel of flows, reached
here through tufrg_loops_noalloc): its error against the FP64 loops, over temperatures and both channels, is no larger."""
import ctypes as C

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1710_08830_gb300 import inputs  # noqa: E402


def _whole_mesh(m, T):
    from paper_1710_08830_gb300 import _lib
    ff = np.ascontiguousarray(m.spec.ff_R, np.int32)
    E, U = m.bands()
    out = torch.zeros(m.loop_shape(), dtype=torch.complex128, device="cuda")
    st = _lib.lib().tufrg_loops_noalloc(m.spec.Lq, m.spec.nc, C.c_void_p(E.data_ptr()), C.c_void_p(U.data_ptr()), C.c_double(m.mu),
                                        C.c_double(T), ff.shape[0], ff.ctypes.data, 3, C.c_void_p(out.data_ptr()),
                                        C.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert st == 0
    return out


@pytest.mark.parametrize("model,Lq,nc,n_ff", [("rashba", 24, 8, 9), ("hubbard", 8, 16, 5), ("rashba", 12, 8, 9), ("hubbard", 20, 9, 9)])
def test_error_is_no_larger_than_the_whole_mesh_sums(model, Lq, nc, n_ff):
    from paper_1710_08830_gb300 import api
    spec = (inputs.rashba_hubbard(1.0, -0.2, 0.3, 2.5, -0.818, Lq=Lq, nc=nc, n_ff=n_ff) if model == "rashba" else
            inputs.hubbard_square(1.0, -0.25, 3.0, filling=0.9, Lq=Lq, nc=nc, n_ff=n_ff))
    m = api.Model(spec, api.SPLIT32)
    exact = api.Model(spec, api.FP64, mu=m.mu)
    half = whole = 0.0
    for T in (0.05, 0.1, 0.2, 0.4, 0.8, 1.6, 3.2):
        ref = exact.loops(T)
        for ch in (0, 1):
            size = float(ref[ch].norm())
            half += (float((m.loops(T)[ch] - ref[ch]).norm()) / size) ** 2
            whole += (float((_whole_mesh(m, T)[ch] - ref[ch]).norm()) / size) ** 2
    print("rms error, half and whole mesh: %.2e %.2e" % ((half / 14) ** 0.5, (whole / 14) ** 0.5))
    assert half <= whole
