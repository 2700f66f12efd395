"""Settings that choose between launches, seen in the kernel timer's counts."""
import pytest
import torch

from paper_2302_07804_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hl():
    from paper_2302_07804_gb300 import henry
    henry.lib()
    torch.cuda.set_device(0)
    return henry


def _launches(s, kind, call):
    s.profile(True)
    call()
    return s.profile_read()[kind][1]


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("level", [0, 1, 2])
def test_batch_limit_of_the_tail_acts_in_both_precisions(hl, precision, level):
    """mg_tail_batch_cells below the smallest batch's cells: no tail, with the
    default mg_tail_cells as with a stated one; the values stay the same."""
    xi = torch.as_tensor(inputs.uniform_xi(7700, 2), device="cuda")
    q = []
    for kw, tail in (({}, True), ({"mg_tail_batch_cells": 1}, False), ({"mg_tail_batch_cells": 0}, True),
                     ({"mg_tail_batch_cells": 1, "mg_tail_cells": 128}, False)):
        s = hl.Solver(precision=precision, fused_small_grids=0, steps0=2, T=720.0, **kw)
        n = _launches(s, "mg_tail", lambda: q.append(s.level_batch_solve(level, xi)[0]))
        s.close()
        assert (n > 0) == tail, kw
    assert all(torch.equal(q[0], v) for v in q[1:])


@pytest.mark.parametrize("precision", [0, 1])
def test_autotuner_times_every_cta_size_that_differs_from_the_default(hl, precision):
    """mg_threads = 0 means 256 threads with FP32 linear algebra, but smaller CTAs
    for small FP64 launches: 256 is a candidate of its own there.  Counted by
    the trials' QoI launches (the same number each) against a configuration
    that states 256, whose candidates are the three other sizes."""
    xi = torch.as_tensor(inputs.uniform_xi(7800, 2), device="cuda")
    n = []
    for threads in (0, 256):
        s = hl.Solver(precision=precision, fused_small_grids=0, steps0=2, T=720.0, mg_threads=threads)
        one = _launches(s, "qoi", lambda: s.level_batch_solve(1, xi))
        n.append(_launches(s, "qoi", lambda: s.autotune(1, xi)) / one)
        s.close()
    assert n[0] - n[1] == (1 if precision == 0 else 0)
