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


def hub_system(n):
    """n - 1 rows coupled to the last one alone: in natural order two phases, the second a single long row."""
    i = np.arange(n - 1, dtype=np.int32)
    rowptr = np.concatenate([2 * np.arange(n, dtype=np.int32), [2 * (n - 1) + n]]).astype(np.int32)
    colidx = np.concatenate([np.stack([i, np.full_like(i, n - 1)], 1).ravel(), np.arange(n, dtype=np.int32)])
    rng = np.random.default_rng(n)
    vals = rng.uniform(-1e-3, 1e-3, (len(colidx), 9))
    rows = np.repeat(np.arange(n), np.diff(rowptr))
    vals[rows == colidx] += 10.0 * np.eye(3).ravel()
    vals[-1] += 1e-2 * n * np.eye(3).ravel()
    return rowptr, colidx, vals


@pytest.mark.parametrize("case", ["long_row", "short_limit"])
def test_own_work_is_no_timeout(case):
    """A limit shorter than a stage's own work: the launches per phase have none, and AUTO takes neither a row of
    tens of thousands of dependent steps nor a limit of a microsecond for an expired wait."""
    if case == "long_row":
        rp, ci, vals = hub_system(20_000)
    else:
        s = synth.config2()
        rp, ci, vals = s.rowptr, s.colidx, s.vals
    nb = len(rp) - 1
    b = torch.ones(3 * nb, dtype=torch.float64, device="cuda")
    got = []
    for sweep, limit in (("per_phase", 0), ("auto", 1 if case == "short_limit" else 1000)):
        o = opm.opm_options_default(sweep_launch=sweep, spin_limit_us=limit,
                                    schedule="natural" if case == "long_row" else "auto")
        st, h = opm.opm_bsr_create(nb, rp, ci, vals, o, check=False)
        assert st == opm.OPM_OK
        x = torch.empty_like(b)
        got.append((opm.opm_bicgstab_solve(h, b, x, rtol=1e-6), x))
        opm.opm_destroy(h)
    assert got[0][0][0] == opm.OPM_OK and got[1][0] == got[0][0] and torch.equal(got[1][1], got[0][1])
