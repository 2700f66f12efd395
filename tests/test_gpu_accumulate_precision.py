"""mlmc_accumulate's centred sum of squares M2 on data whose mean is large
against their spread, against the oracle's two-pass moments.

Bound, fixed beforehand: the values' distances from a pivot within a factor two
of them are exact, so what is left are R roundings of a sum's chain - the rows a
lane adds, 5 of its warp, 8 warps, 8 CTAs and the merge: R = rows a lane + 30 -
on the sums of (y - k)^2 and of y - k, three of them in all, times the at most
four-fold cancellation of M2 = s2 - s1^2 / n that the kernel accepts: 12 R u with
u = 2^-53.  The oracle takes each column by itself, contiguous and less its first
value (an exact difference on these inputs), so that its sums run pairwise over
values of the spread's size and its own error is a few u; over rows of 1e8 its
mean alone would leave 2e-12.
"""
import numpy as np
import pytest
import torch

from oracle import mlmc as omlmc
from paper_2302_07804_gb300 import inputs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module")
def hl():
    from paper_2302_07804_gb300 import henry
    henry.lib()
    torch.cuda.set_device(0)
    return henry


def _shape(n, n_qoi):
    """Columns a CTA takes, its rows a step and the CTAs of a cluster."""
    cw = 16
    while cw > 1 and (n_qoi + cw - 1) // cw < 16:
        cw //= 2
    return cw, 256 // cw, max(1, min(8, -(-n // (512 // cw))))


def _check(hl, qf, qc, status):
    n, n_qoi = qf.shape
    _, rows, ctas = _shape(n, n_qoi)
    tol = 12 * (-(-n // (rows * ctas)) + 30) * 2.0 ** -53
    dev = [None if a is None else torch.as_tensor(a, device=DEV) for a in (qf, qc, status)]
    sums = torch.zeros((2, n_qoi, 3), dtype=torch.float64, device=DEV)
    hl.mlmc_accumulate(1, dev[0], dev[1], dev[2], sums)
    keep = np.ones(n, dtype=bool) if status is None else status == 0
    y = omlmc.level_differences(qf[keep], None if qc is None else qc[keep])
    for got, v in zip(sums.cpu().numpy(), (y, qf[keep])):
        for k in range(n_qoi):
            col = np.ascontiguousarray(v[:, k])
            m, mean, m2 = omlmc.two_pass_moments(col - col[0])
            assert got[k, 0] == m
            np.testing.assert_allclose(got[k, 1], col[0] + mean, rtol=0, atol=1e-13 * np.abs(v).max())
            np.testing.assert_allclose(got[k, 2], m2, rtol=tol, atol=0)


@pytest.mark.parametrize("n,n_qoi", [(513, 2), (20011, 2), (4099, 33), (20011, 257)])
@pytest.mark.parametrize("mean,sd", [(1.0e8, 1.0), (0.999, 1.0e-8)])
def test_spread_far_below_the_mean(hl, n, n_qoi, mean, sd):
    gen = inputs.rng(7300 + n + n_qoi)
    qf = mean + sd * gen.standard_normal((n, n_qoi))
    qc = 0.25 * mean + sd * gen.standard_normal((n, n_qoi))
    _check(hl, qf, None, None)
    _check(hl, qf, qc, (gen.random(n) < 0.2).astype(np.int32))
@pytest.mark.parametrize("n,n_qoi", [(100, 2), (513, 1), (20011, 2), (20011, 33), (20011, 257)])
@pytest.mark.parametrize("head", [8, 16, "every", "outlier"])
def test_first_rows_failed_or_far_from_the_rest(hl, n, n_qoi, head):
    """The first rows of a CTA's share, which place the pivot, have failed (the
    first 8 or 16 of the batch, or 8 of every step) or lie far from the rest."""
    gen = inputs.rng(7400 + n + n_qoi)
    qf = 0.999 + 1.0e-8 * gen.standard_normal((n, n_qoi))
    qc = 0.25 + 1.0e-8 * gen.standard_normal((n, n_qoi))
    _, rows, ctas = _shape(n, n_qoi)
    status = np.zeros(n, dtype=np.int32)
    if head == "every":
        status[np.arange(n) % rows < 8] = 1
    elif head == "outlier":  # one used row among each CTA's first 8, 1e4 standard deviations off
        for r in range(ctas):
            status[r * rows + 1:r * rows + 8] = 1
            qf[r * rows] += 1.0e-4 * (1.0 + 0.1 * r)
    else:
        status[:head] = 1
    _check(hl, qf, None, status)
    _check(hl, qf, qc, status)


def test_one_used_row_behind_failed_ones(hl):
    qf = 0.999 + 1.0e-8 * inputs.rng(7500).standard_normal((100, 3))
    status = np.ones(100, dtype=np.int32)
    status[99] = 0
    sums = torch.zeros((2, 3, 3), dtype=torch.float64, device=DEV)
    hl.mlmc_accumulate(1, torch.as_tensor(qf, device=DEV), None, torch.as_tensor(status, device=DEV), sums)
    S = sums.cpu().numpy()
    assert np.all(S[:, :, 0] == 1) and np.all(S[:, :, 1] == qf[99]) and np.all(S[:, :, 2] == 0.0)
