"""Which calls go to the resident kernel, and what they report."""
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
