"""The resident kernel (one cooperative launch per refactorisation and solve:
sweep_launch "auto" on a single system) against the launches per phase: the
same arithmetic in the same order, so factors, solutions, iteration counts
and residuals are compared bitwise, at the edges of its units (32-row slices,
256- and 1024-row tiles, 8,192-row groups) and of its two forms."""
import numpy as np
import pytest

from paper_2309_11488_gb300 import opm, synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def grid(nx, ny, nz, seed=3):
    logk = np.random.default_rng(seed).normal(size=(nz, ny, nx))
    return synth.grid_system(nx, ny, nz, logk, seed=synth.SEED_BASE + seed)


def both_forms(s, precision, rtol, schedule="auto", part=None, wells=None, reuse=0, refactor=True):
    """(factors, x, status, iters, relres) with launches per phase and resident."""
    b = dev(s.x_true)  # any right-hand side does
    vals2 = dev(s.vals * (1.0 + 0.01 * np.cos(np.arange(s.nnzb)))[:, None])
    out = []
    for sweep in ("per_phase", "auto"):
        with opm.Solver(s.nb, dev(s.rowptr), dev(s.colidx), dev(s.vals), schedule=schedule, precision=precision,
                        sweep_launch=sweep, part=part, product_reuse=reuse) as sv:
            if wells is not None:
                assert sv.set_wells(wells) == opm.OPM_OK
            x = torch.full_like(b, 7.0)
            if refactor:
                sv.launch(vals2, b, x, rtol=rtol)
                st, it, rr = sv.wait()
            else:
                _, st, it, rr = sv.solve(b, x, rtol=rtol)
            x2, st2, it2, rr2 = sv.solve(b, rtol=1e-2, maxit=3)  # again, on the kept factors
            out.append((*sv.factors(), x.cpu().numpy(), x2.cpu().numpy(), np.array([st, it, rr, st2, it2, rr2])))
    for a, c in zip(*out):
        np.testing.assert_array_equal(a, c)
    assert out[0][-1][0] == 0


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("n", [1, 31, 32, 33, 255, 257, 1023, 1025, 8191, 8193])
def test_edges_of_units(n, precision):
    both_forms(synth.chain_system(n), precision, 1e-8, schedule="colour")


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("dims", [(39, 39, 40), (41, 39, 40), (68, 67, 68), (69, 67, 68)])
def test_edges_of_forms(dims, precision):
    # 60,800 rows: the last size of the three-warp form on 152 SMs; 311,296: the last of the resident kernel
    both_forms(grid(*dims), precision, 1e-3)


@pytest.mark.parametrize("schedule", ["natural", "level", "colour", "colour_kempe"])
def test_schedules_and_long_rows(schedule):
    # rows past the blocks loaded ahead, non-symmetric pattern; long dependency chains in natural order
    s = synth.one_way_system(synth.random_pattern_system(700, 9, 11), 0.3, 12)
    both_forms(s, "fp64", 1e-10, schedule=schedule)


@pytest.mark.parametrize("n", [14, 42])  # three-warp and one-warp form
@pytest.mark.parametrize("case", ["jacobi_wells", "wells", "plain_product", "solve_only"])
def test_options(n, case):
    s = synth.config3(n)
    part = synth.partition_grid(s, 5) if case == "jacobi_wells" else None
    wells = synth.wells(s, 9, 4) if "wells" in case else None
    both_forms(s, "fp64", 1e-6, part=part, wells=wells, reuse=-1 if case == "plain_product" else 0,
               refactor=case != "solve_only")


def test_bounded_wait_expires_and_singular_pivot():
    s = synth.config2()
    st, h = opm.opm_bsr_create(s.nb, s.rowptr, s.colidx, s.vals,
                               opm.opm_options_default(spin_limit_us=20000, debug_skip_item=3), check=False)
    assert st == opm.OPM_ERR_TIMEOUT
    opm.opm_destroy(h)
    rows = np.repeat(np.arange(s.nb), np.diff(s.rowptr))
    bad = s.vals.copy()
    bad[np.flatnonzero(rows == s.colidx)[5]] = 0.0
    b = dev(s.x_true)
    with opm.Solver(s.nb, dev(s.rowptr), dev(s.colidx), dev(s.vals)) as sv:
        x0, st0, it0, rr0 = sv.solve(b)
        x = torch.empty_like(b)
        sv.launch(dev(bad), b, x)
        st, it, rr = sv.wait()
        assert st == opm.OPM_ERR_ZERO_PIVOT and (x == 0).all() and np.isnan(rr)
        assert sv.factor(dev(bad)) == opm.OPM_ERR_ZERO_PIVOT and opm.opm_last_error_row(sv.h) == 5
        assert sv.factor(dev(s.vals)) == opm.OPM_OK  # recovers
        x1, st1, it1, rr1 = sv.solve(b)
        assert (st1, it1, rr1) == (st0, it0, rr0) and torch.equal(x1, x0)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("n", [8, 14, 42, 70])  # three-warp, one-warp form, launches per phase
def test_operators_alone_and_in_place(n, precision):
    """Product and application against the launches per phase, also with the output over the input (at an offset
    too), and a solve whose x takes b's place."""
    s = synth.config3(n)
    x = dev(s.x_true)
    n3 = x.numel()
    out = []
    for sweep in ("per_phase", "auto"):
        with opm.Solver(s.nb, dev(s.rowptr), dev(s.colidx), dev(s.vals), precision=precision, sweep_launch=sweep) as sv:
            y, z = sv.spmv(x), sv.ilu_apply(x)
            for op, ref in ((sv.spmv, y), (sv.ilu_apply, z)):
                for shift in (0, 3):
                    buf = torch.zeros(n3 + 3, dtype=torch.float64, device="cuda")
                    buf[:n3] = x
                    assert torch.equal(op(buf[:n3], buf[shift:shift + n3]), ref)
            a, st, it, rr = sv.solve(y, rtol=1e-4)
            b = y.clone()
            a2, st2, it2, rr2 = sv.solve(b, b, rtol=1e-4)
            assert (st, it, rr) == (st2, it2, rr2) and torch.equal(a, a2)
            out.append((y, z, a))
    for u, v in zip(*out):
        assert torch.equal(u, v)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("dims", [(33, 1, 1), (20, 20, 20), (32, 30, 19), (32, 571, 1)])
def test_handles_on_streams_of_their_own(dims, precision):
    """Three handles refactor and solve at once, each on a stream of its own, which bounds the resident kernel's grid
    and sizes (18,240 rows: the last on 152 SMs): the bits of the launches per phase on the default stream."""
    s = grid(*dims)
    vals = [dev(s.vals * (1.0 + 0.01 * k * np.cos(np.arange(s.nnzb)))[:, None]) for k in range(3)]
    b = dev(s.x_true)
    an = opm.Analysis(s.nb, s.rowptr, s.colidx)
    want = []
    for v in vals:
        with opm.Solver.from_analysis(an, v, precision=precision, sweep_launch="per_phase") as sv:
            want.append((*sv.solve(b, rtol=1e-3), sv.ilu_apply(b)))
    streams = [torch.cuda.Stream() for _ in vals]
    torch.cuda.synchronize()
    sv = [opm.Solver.from_analysis(an, vals[0], precision=precision, stream=q) for q in streams]
    xs = [torch.empty_like(b) for _ in vals]
    torch.cuda.synchronize()
    for h, v, x in zip(sv, vals, xs):
        h.launch(v, b, x, rtol=1e-3)
    for h, x, (xw, st, it, rr, z) in zip(sv, xs, want):
        assert h.wait() == (st, it, rr) and torch.equal(x, xw)
        out = torch.empty_like(b)
        torch.cuda.synchronize()
        h.ilu_apply(b, out)
        assert torch.equal(out, z)
        h.close()
