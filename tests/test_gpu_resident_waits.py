"""Bounded waits of the resident kernel: what a call returns and leaves behind when one expires."""
import ctypes

import numpy as np
import pytest

from paper_2309_11488_gb300 import opm, synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def short_wait_batch(h):
    """A batch of the handle alone, whose launches lack the arrivals of one CTA."""
    b = opm.Batch([h])
    opm.lib().opm_batch_destroy(ctypes.c_void_p(b.ptr))
    o = opm.opm_options_default(spin_limit_us=20000, debug_skip_item=3)
    out = ctypes.c_void_p()
    hs = (ctypes.c_void_p * 1)(h.ptr)
    assert opm.lib().opm_batch_create(1, hs, ctypes.byref(o), ctypes.byref(out)) == opm.OPM_OK
    b.ptr = out.value
    return b


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("n", [36, 42])  # three-warp and one-warp form
def test_expired_wait_zeroes_x_and_leaves_no_factors(n, precision):
    s = synth.config3(n)
    b = dev(s.x_true)
    vals = dev(s.vals)
    with opm.Solver(s.nb, dev(s.rowptr), dev(s.colidx), vals, precision=precision) as sv:
        want = sv.solve(b, rtol=1e-4)
        z = sv.ilu_apply(b)
        short = short_wait_batch(sv.h)
        # a solve that runs out: x is zero, the factors stay
        x = torch.full_like(b, 7.0)
        short.launch(None, [b], [x])
        st, each, _, rr = short.wait()
        assert st == opm.OPM_ERR_TIMEOUT and each == [st] and (x == 0).all() and np.isnan(rr[0])
        assert torch.equal(sv.ilu_apply(b), z)
        # a refactorisation that runs out: x is zero, and what needs factors says so
        x = torch.full_like(b, 7.0)
        short.launch([vals], [b], [x])
        assert short.wait()[0] == opm.OPM_ERR_TIMEOUT and (x == 0).all()
        z2 = torch.empty_like(b)
        assert opm.opm_ilu_apply(sv.h, b, z2) == opm.OPM_ERR_TIMEOUT
        x2 = torch.full_like(b, 7.0)
        assert opm.opm_bicgstab_solve(sv.h, b, x2)[0] == opm.OPM_ERR_TIMEOUT and (x2 == 0).all()
        assert sv.gmres(b)[1] == opm.OPM_ERR_TIMEOUT
        # host vectors: the staging vector's zeros, not the last solve's x
        xh = np.full(3 * s.nb, 7.0)
        assert opm.opm_bicgstab_solve(sv.h, s.x_true, xh)[0] == opm.OPM_ERR_TIMEOUT and (xh == 0).all()
        short.close()
        # and all is as before after the next factorisation
        assert sv.factor(vals) == opm.OPM_OK
        got = sv.solve(b, rtol=1e-4)
        assert got[1:] == want[1:] and torch.equal(got[0], want[0]) and torch.equal(sv.ilu_apply(b), z)
