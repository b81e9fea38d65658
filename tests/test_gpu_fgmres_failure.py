"""A solve that a CUDA call of its own ends: what the caller is told."""
import ctypes as C

import numpy as np
import pytest

import abilu_inputs as gen


@pytest.mark.gpu
@pytest.mark.parametrize("zero_guess", [True, False])
def test_a_failed_solve_reports_its_first_error_and_leaves_the_handle_usable(zero_guess):
    """A solve waits for its stream, so on a stream under capture CUDA refuses the
    wait and nothing runs.  The result holds the returned code, the message names
    the refused step and not a later clean-up, and the next solve finds no error
    left over."""
    import torch
    import paper_1912_00539_gb300.abilu as ab
    s = gen.small_system(20, 10, seed=1)
    pat = ab.Pattern(torch.from_numpy(s.rowptr).cuda(), torch.from_numpy(s.colind).cuda())
    A, b = torch.from_numpy(s.vals).cuda(), torch.from_numpy(s.b).cuda()
    fac, x = ab.Factors(pat, "f32"), torch.zeros_like(b)
    opts = dict(build_sweeps=3, apply_sweeps_lower=2, apply_sweeps_upper=2, mode="sync", zero_guess=zero_guess)
    good = ab.fgmres_solve(pat, A, fac, b, x, **opts)   # the handle's workspace and events exist
    x0 = x.clone()
    drv = C.CDLL("libcuda.so.1")
    st = torch.cuda.Stream()
    torch.cuda.synchronize()
    o, r, g = ab.default_opts(), ab.FgmresResult(), C.c_void_p()
    o.zero_guess, r.status = int(zero_guess), -99
    assert drv.cuStreamBeginCapture_v2(C.c_void_p(st.cuda_stream), 2) == 0
    code = ab._lib.fgmres_solve(pat.handle, C.c_void_p(A.data_ptr()), fac.handle, C.c_void_p(b.data_ptr()),
                                C.c_void_p(x.data_ptr()), C.byref(o), C.byref(r), C.c_void_p(st.cuda_stream))
    text = ab._lib.abilu_last_error().decode()
    drv.cuStreamEndCapture(C.c_void_p(st.cuda_stream), C.byref(g))
    if g.value:
        drv.cuGraphDestroy(g)
    assert code not in (ab.OK, ab.WARN_SINGULAR, ab.ENOCONV) and r.status == code
    assert text.startswith("fgmres") and "zero" not in text and "Memset" not in text, text
    torch.cuda.synchronize()
    assert torch.equal(x, x0)   # nothing ran
    x.zero_()
    again = ab.fgmres_solve(pat, A, fac, b, x, **opts)
    assert again.converged and again.iters == good.iters
    assert np.array_equal(x.cpu().numpy(), x0.cpu().numpy())
