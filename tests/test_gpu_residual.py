"""opm_bsr_residual_noalloc at the edges of its units (10-row groups, 40-row
CTAs, 72-block chunks, several groups per warp) and for rows that do not
follow one another, against the product in plain PyTorch."""
import numpy as np
import pytest

from paper_2309_11488_gb300 import opm, synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def check(rowptr, colidx, vals, nb, want=opm.OPM_OK, fault_row=None):
    rng = np.random.default_rng(nb)
    x, b = dev(rng.uniform(-1, 1, 3 * nb)), dev(rng.uniform(-1, 1, 3 * nb))
    r, norms = torch.full_like(x, np.nan), torch.zeros(2, dtype=torch.float64, device="cuda")
    for _ in range(2):  # the scratch words are zero again after a call
        assert opm.opm_bsr_residual_noalloc(nb, dev(rowptr), dev(colidx), dev(vals), x, b, r, norms) == want
    lens = np.diff(rowptr).clip(min=0)
    rows = np.repeat(np.arange(nb), lens)
    m = np.concatenate([np.arange(a, a + k) for a, k in zip(rowptr[:-1], lens)]) if len(rows) else rows
    cols = colidx[m]
    ok = (cols >= 0) & (cols < nb)
    prod = (dev(vals[m[ok]]).view(-1, 3, 3) * x.view(-1, 3)[dev(cols[ok].astype(np.int64))].unsqueeze(1)).sum(2)
    y = torch.zeros(nb, 3, dtype=torch.float64, device="cuda").index_add_(0, dev(rows[ok]), prod)
    size = torch.zeros(nb, 3, dtype=torch.float64, device="cuda").index_add_(0, dev(rows[ok]), prod.abs())
    ref = b - y.view(-1)
    # a row's rounding errors, at most one unit per operation, against the sum of its terms' sizes
    bound = 1e-15 * (3 + 3 * lens.max()) * (size.view(-1) + b.abs()) * (1 + x.abs().max())
    assert ((r - ref).abs() <= bound).all()
    if want == opm.OPM_OK:
        torch.testing.assert_close(norms, torch.stack([ref.norm(), b.norm()]), rtol=1e-12, atol=0)
    else:
        assert torch.isnan(norms).all()


@pytest.mark.parametrize("nb", [1, 9, 10, 11, 39, 41, 3001])
def test_edges(nb):
    s = synth.random_pattern_system(nb, 5, nb) if nb > 1 else synth.block_diagonal_system(1, 3)
    check(s.rowptr, s.colidx, s.vals, nb)


def test_long_rows_and_several_groups_per_warp():
    s = synth.random_pattern_system(90, 1, 5, dense=True)  # 90 blocks a row: more than a chunk
    check(s.rowptr, s.colidx, s.vals, s.nb)
    s = synth.chain_system(330_000)  # several groups per warp
    check(s.rowptr, s.colidx, s.vals, s.nb)


def test_rows_out_of_order_and_columns_outside():
    s = synth.random_pattern_system(400, 4, 9)
    rp = s.rowptr.copy()
    rp[200] = rp[201] + 3  # row 199 runs on into the next rows, row 200 ends before its start
    check(rp, s.colidx, s.vals, s.nb, want=opm.OPM_ERR_PATTERN)
    ci = s.colidx.copy()
    ci[[5, 700]] = [s.nb, -1]
    check(s.rowptr, ci, s.vals, s.nb, want=opm.OPM_ERR_PATTERN)
