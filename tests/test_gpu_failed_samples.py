"""What a failed sample's outputs hold."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hl():
    from paper_2302_07804_gb300 import henry
    henry.lib()
    torch.cuda.set_device(0)
    return henry


@pytest.mark.parametrize("precision,K", [(0, 9.0e299), (1, 1.0e40)])
@pytest.mark.parametrize("level,with_coarse", [(0, False), (1, True)])
def test_non_finite_newton_step_leaves_no_finite_qoi(hl, precision, K, level, with_coarse):
    """A permeability whose Jacobian overflows the linear algebra's type while
    the residual does not (hardly any gravity): the Newton step is NaN, the
    sample fails as non-finite and its QoIs are NaN, not the last state's."""
    s = hl.Solver(precision=precision, K_mean=K, g=1e-305 if precision == 0 else 1e-100, fused_small_grids=0,
                  newton_maxit=4)
    xi = torch.zeros((3, 3), dtype=torch.float64, device="cuda")
    qf, qc, st, _ = s.level_batch_solve(level, xi, with_coarse=with_coarse, allow_failures=True)
    s.close()
    assert bool((st == 3).all())
    assert bool(torch.isnan(qf).all())
    assert qc is None or bool(torch.isnan(qc).all())
