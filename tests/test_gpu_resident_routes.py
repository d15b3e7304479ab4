"""Which calls go to the resident kernel, and what they report."""
import ctypes

import numpy as np
import pytest

from paper_2309_11488_gb300 import opm, synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def test_launches_are_counted():
    """opm_timing.launches of the resident form: one per factorisation (the handle's first too), solve, or both."""
    s = synth.config1()
    b = dev(s.x_true)
    with opm.Solver(s.nb, dev(s.rowptr), dev(s.colidx), dev(s.vals)) as sv:
        seen = [sv.timing().launches]
        for call in (lambda: sv.factor(dev(s.vals)), lambda: sv.solve(b), lambda: sv.ilu_apply(b),
                     lambda: (sv.launch(dev(s.vals), b, torch.empty_like(b)), sv.wait())):
            call()
            seen.append(sv.timing().launches)
        assert seen == [1, 2, 3, 4, 5]


def flat(nx, ny):
    return synth.grid_system(nx, ny, 1, np.random.default_rng(1).normal(size=(1, ny, nx)), seed=3)


# (system, schedule, partitions, precision): whether the resident kernel refactors and solves it, solves it on kept
# factors, and applies it alone; by phases
ROUTES = [
    (lambda: synth.config3(14), "level", 0, "fp64", True, True, True),  # 47 phases, trios
    (lambda: synth.config3(14), "level", 0, "fp32", True, True, False),
    (lambda: synth.config3(14), "auto", 0, "fp32", True, True, True),
    (lambda: synth.chain_system(192), "natural", 0, "fp64", True, True, True),
    (lambda: synth.chain_system(193), "natural", 0, "fp64", True, False, False),
    (lambda: flat(200, 15), "level", 0, "fp32", True, False, False),  # 214 phases
    (lambda: synth.chain_system(1025), "natural", 0, "fp32", True, True, True),  # more than launches are made for
    (lambda: synth.config3(45), "auto", 0, "fp64", True, True, True),  # 3 phases, a warp per slice
    (lambda: synth.config3(45), "level", 512, "fp64", False, False, False),  # 22 phases
]


@pytest.mark.parametrize("make, schedule, parts, precision, steps, solves, applies", ROUTES)
@pytest.mark.parametrize("nwells", [0, 2])
def test_routes_by_phases(make, schedule, parts, precision, steps, solves, applies, nwells):
    """A route is seen in the kernels that a call launches; the bits are those of the launches per phase, also when
    wells come and go between calls."""
    s = make()
    part = np.ascontiguousarray(synth.partition_grid(s, parts), dtype=np.int32) if parts else None
    if nwells and s.nb < 2000:
        pytest.skip("wells are placed on grids")
    b, v = dev(s.x_true), dev(s.vals)
    out = []
    for sweep in ("per_phase", "auto"):
        with opm.Solver(s.nb, dev(s.rowptr), dev(s.colidx), v, schedule=schedule, precision=precision, part=part,
                        sweep_launch=sweep) as sv:
            x = torch.empty_like(b)
            got, n = [], [sv.timing().launches]
            if nwells:
                assert sv.set_wells(synth.wells(s, nwells, 4)) == opm.OPM_OK
            sv.launch(v, b, x, rtol=1e-4)
            got += [sv.wait(), x]
            n.append(sv.timing().launches)
            got += sv.solve(b, rtol=1e-4)
            n.append(sv.timing().launches)
            got.append(sv.ilu_apply(b))
            n.append(sv.timing().launches)
            if nwells:
                assert sv.set_wells(None) == opm.OPM_OK
                got += sv.solve(b, rtol=1e-4)
            out.append(got)
    assert [k == 1 for k in np.diff(n)] == [steps, solves, applies]
    for p, q in zip(*out):
        assert torch.equal(p, q) if torch.is_tensor(p) else p == q


def test_edges_of_the_three_warp_form():
    """On both sides of the last size of the three-warp form, on all SMs, with up to 2.5 slices per trio; and the
    44,431-row mesh.  The limit follows from the number of SMs."""
    slices = 5 * 5 * torch.cuda.get_device_properties(0).multi_processor_count // 2
    side = round((32 * slices) ** 0.5 / 8) * 8
    systems = [synth.config2()]
    for rows in (32 * slices, 32 * slices + 1):  # chains: any row count
        systems.append(synth.chain_system(rows))
    systems.append(flat(side, 32 * slices // side))
    for s in systems:
        for precision in ("fp64", "fp32"):
            b, v = dev(s.x_true), dev(s.vals)
            out = []
            for sweep in ("per_phase", "auto"):
                with opm.Solver(s.nb, dev(s.rowptr), dev(s.colidx), v, precision=precision, sweep_launch=sweep) as sv:
                    x = torch.empty_like(b)
                    sv.launch(v, b, x, rtol=1e-6)
                    out.append((sv.wait(), x, sv.ilu_apply(b), *map(torch.from_numpy, sv.factors())))
            assert out[0][0] == out[1][0]
            assert all(torch.equal(p, q) for p, q in zip(out[0][1:], out[1][1:]))


def test_sizes_on_a_stream_of_its_own():
    """A quarter of the SMs: two slices per trio for two phases, three for more."""
    trios = 5 * ((torch.cuda.get_device_properties(0).multi_processor_count + 3) // 4)
    side = torch.cuda.Stream()
    for make, resident in ((lambda: synth.chain_system(64 * trios), True), (lambda: synth.chain_system(64 * trios + 1), False),
                           (lambda: synth.config3(26), 521 <= 3 * trios)):  # 16,667 rows, 3 phases
        s = make()
        b, v = dev(s.x_true), dev(s.vals)
        x = torch.empty_like(b)
        torch.cuda.synchronize()
        with opm.Solver(s.nb, dev(s.rowptr), dev(s.colidx), v, stream=side) as sv:
            n0 = sv.timing().launches
            sv.launch(v, b, x)
            assert sv.wait()[0] == opm.OPM_OK
            assert (sv.timing().launches - n0 == 1) == resident


def test_legacy_stream_by_name():
    """cudaStreamLegacy is the default stream: 44,431 rows are one launch there, and not on a stream of their own."""
    s = synth.config2()
    b, v = dev(s.x_true), dev(s.vals)
    torch.cuda.synchronize()
    for stream, resident in ((1, True), (torch.cuda.Stream(), False)):
        with opm.Solver(s.nb, dev(s.rowptr), dev(s.colidx), v, stream=stream) as sv:
            n0 = sv.timing().launches
            assert sv.solve(b)[1] == opm.OPM_OK
            assert (sv.timing().launches - n0 == 1) == resident


def test_batch_of_one_that_sits_out():
    s = synth.config1()
    b, v = dev(s.x_true), dev(s.vals)
    with opm.Solver(s.nb, dev(s.rowptr), dev(s.colidx), v) as sv, opm.Batch([sv.h]) as one:
        want = sv.solve(b)
        one.launch([None], [None], [None])
        assert one.wait() == (opm.OPM_OK, [opm.OPM_OK], [0], [0.0])
        x = torch.empty_like(b)
        one.launch([v], [b], [x])
        assert one.wait()[0] == opm.OPM_OK and torch.equal(x, want[0])


def test_stream_with_a_part_of_the_device():
    """A green context of 16 SMs cannot hold a quarter of the device's CTAs at once: the launches per phase."""
    cu = ctypes.CDLL("libcuda.so.1")
    if not hasattr(cu, "cuGreenCtxStreamCreate"):
        pytest.skip("this driver has no green contexts")
    torch.zeros(1, device="cuda")
    device, whole, part = ctypes.c_int(), ctypes.create_string_buffer(144), ctypes.create_string_buffer(144)
    groups, desc, ctx, stream = ctypes.c_uint(1), ctypes.c_void_p(), ctypes.c_void_p(), ctypes.c_void_p()
    assert cu.cuDeviceGet(ctypes.byref(device), 0) == 0
    assert cu.cuDeviceGetDevResource(device, whole, 1) == 0  # CU_DEV_RESOURCE_TYPE_SM
    assert cu.cuDevSmResourceSplitByCount(part, ctypes.byref(groups), whole, None, 0, 16) == 0
    assert cu.cuDevResourceGenerateDesc(ctypes.byref(desc), part, 1) == 0
    assert cu.cuGreenCtxCreate(ctypes.byref(ctx), desc, device, 1) == 0  # CU_GREEN_CTX_DEFAULT_STREAM
    assert cu.cuGreenCtxStreamCreate(ctypes.byref(stream), ctx, 1, 0) == 0  # CU_STREAM_NON_BLOCKING
    try:
        s = synth.config3(14)
        b, v = dev(s.x_true), dev(s.vals)
        torch.cuda.synchronize()
        out = []
        for where in (None, stream.value):
            with opm.Solver(s.nb, dev(s.rowptr), dev(s.colidx), v, stream=where) as sv:
                x, z = torch.empty_like(b), torch.empty_like(b)
                torch.cuda.synchronize()
                sv.launch(v, b, x, rtol=1e-6)
                out.append((sv.wait(), x, sv.ilu_apply(b, z)))
        assert out[0][0] == out[1][0] and torch.equal(out[0][1], out[1][1]) and torch.equal(out[0][2], out[1][2])
    finally:
        torch.cuda.synchronize()
        cu.cuStreamDestroy_v2(stream)
        cu.cuGreenCtxDestroy(ctx)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("big", [8, 32, 70])  # rows past the resident kernel's sizes with 70: two orders of summation
def test_batches_have_the_bits_of_each_alone(big, precision):
    systems = [synth.config3(big), synth.config1(), synth.chain_system(33)]
    b, v = [dev(s.x_true) for s in systems], [dev(s.vals) for s in systems]
    sv = [opm.Solver(s.nb, dev(s.rowptr), dev(s.colidx), a, precision=precision) for s, a in zip(systems, v)]
    alone = [h.solve(c, rtol=1e-4) for h, c in zip(sv, b)]
    with opm.Batch([h.h for h in sv]) as batch:
        x = [torch.empty_like(c) for c in b]
        batch.launch(v, b, x, rtol=1e-4)
        st, each, iters, relres = batch.wait()
    assert st == opm.OPM_OK
    for k, (xa, sa, ia, ra) in enumerate(alone):
        assert (each[k], iters[k], relres[k]) == (sa, ia, ra) and torch.equal(x[k], xa)
    for h in sv:
        h.close()
