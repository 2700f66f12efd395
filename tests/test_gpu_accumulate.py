"""mlmc_accumulate at the sizes where its column groups (1 .. 16 QoIs), warp
steps and clusters of CTAs change, against the oracle's two-pass moments.

Tolerances, fixed beforehand: a lane sums at most n / 512 + 16 values about a
pivot inside the data, so its sums are off by at most ~60 roundings (7e-15);
the pivot's distance from the mean costs a factor 1 + (k - mean)^2 / var <= 10
on these inputs, so M2 agrees to relative 1e-12 and the mean to 1e-13 of the
values' size.
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


@pytest.mark.parametrize("n_qoi", [1, 2, 15, 16, 17, 33, 257, 527])
@pytest.mark.parametrize("n", [1, 2, 15, 33, 513, 4099, 20011])
def test_batch_moments_match_two_pass(hl, n, n_qoi):
    if n * n_qoi > 3_000_000:
        n = 3001
    gen = inputs.rng(7100 + n + n_qoi)
    qf = 0.5 + 0.3 * gen.random((n, n_qoi))
    qf[:, 0] *= 200.0
    qc = qf * (1.0 + 0.01 * gen.standard_normal((n, 1)))
    status = (gen.random(n) < 0.2).astype(np.int32)
    dev = [torch.as_tensor(a, device=DEV) for a in (qf, qc, status)]
    for coarse in (True, False):
        for failed in (True, False):
            keep = status == 0 if failed else np.ones(n, dtype=bool)
            sums = torch.zeros((2, n_qoi, 3), dtype=torch.float64, device=DEV)
            hl.mlmc_accumulate(1, dev[0], dev[1] if coarse else None, dev[2] if failed else None, sums)
            S = sums.cpu().numpy()
            y = omlmc.level_differences(qf[keep], qc[keep] if coarse else None)
            for got, v in ((S[0], y), (S[1], qf[keep])):
                m, mean, m2 = omlmc.two_pass_moments(v)
                assert np.all(got[:, 0] == m)
                np.testing.assert_allclose(got[:, 1], mean, rtol=0, atol=1e-13 * max(1.0, np.abs(v).max(initial=0)))
                np.testing.assert_allclose(got[:, 2], m2, rtol=1e-12, atol=1e-26 * max(m, 1))


def test_infinite_values_and_batches_without_samples(hl):
    """An infinite QoI gives an infinite mean and a NaN M2 in its own column; a
    batch with no usable sample leaves the sums as they were."""
    qf = torch.full((600, 3), 0.25, dtype=torch.float64, device=DEV)
    qf[77, 1] = float("inf")
    sums = torch.zeros((2, 3, 3), dtype=torch.float64, device=DEV)
    hl.mlmc_accumulate(0, qf, None, None, sums)
    S = sums.cpu().numpy()
    assert np.all(S[:, :, 0] == 600) and np.all(np.isinf(S[:, 1, 1])) and np.all(np.isnan(S[:, 1, 2]))
    assert np.all(S[:, [0, 2], 1] == 0.25) and np.all(S[:, [0, 2], 2] == 0.0)
    before = sums.clone()
    hl.mlmc_accumulate(0, qf, None, torch.ones(600, dtype=torch.int32, device=DEV), sums)
    assert torch.equal(sums.nan_to_num(7.0), before.nan_to_num(7.0))
