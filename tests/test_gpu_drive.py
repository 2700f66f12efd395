"""How a solve is driven changes no value: the fused multigrid tail from the
fine grid itself, and the captured BiCGStab iterations, against separate kernels
and plain launches, bit for bit, at the sizes and settings where the choice
changes."""
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


def _wedge(n, ny, nx, shift):
    x = ((torch.arange(nx, dtype=torch.float64, device="cuda") + 0.5) * (2.0 / nx))[None, None, :]
    y = ((torch.arange(ny, dtype=torch.float64, device="cuda") + 0.5) / ny)[None, :, None]
    s = torch.linspace(0.0, 0.2, n, dtype=torch.float64, device="cuda")[:, None, None]
    c = 0.5 * (1.0 + torch.tanh((x - 1.3 - 0.5 * y + shift + s) / 0.15))
    p = 1000.0 * 9.81 * (1.0 - y) * (1.0 + 0.025 * c) + 20.0 * torch.cos(3.0 * x + 2.0 * y)
    return torch.stack([p, c], dim=-1).contiguous()


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("level,n", [(0, 1), (0, 152), (0, 153), (0, 1025), (1, 1), (1, 153), (1, 305), (2, 3)])
@pytest.mark.parametrize("nu", [(2, 2), (1, 0), (0, 1)])
def test_default_tail_start_is_bit_identical_to_separate_kernels(hl, precision, level, n, nu):
    if nu != (2, 2) and n > 153:
        n = 2
    ny, nx = 16 << level, 32 << level
    xi = torch.as_tensor(inputs.uniform_xi(9100 + level, n), device="cuda")
    b = torch.as_tensor(inputs.rng(9101 + n).standard_normal((n, ny, nx, 2)), device="cuda")
    z = []
    for tail in (-1, 0):
        s = hl.Solver(precision=precision, mg_tail_cells=tail, nu1=nu[0], nu2=nu[1])
        z.append(s.precondition(level, xi, _wedge(n, ny, nx, 0.0), _wedge(n, ny, nx, 0.02), b))
        s.close()
    assert bool(torch.isfinite(z[0]).all()) and torch.equal(z[0], z[1])


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("res_first,every,maxit", [(-1, 1, 30), (0, 1, 30), (1, 1, 30), (2, 1, 30), (3, 2, 30), (4, 3, 30),
                                                    (5, 1, 30), (9, 1, 30), (-1, 3, 30), (2, 1, 1), (2, 1, 2)])
def test_captured_iterations_equal_plain_launches(hl, precision, res_first, every, maxit):
    xi = torch.as_tensor(inputs.uniform_xi(9200, 5), device="cuda")
    out = []
    for graphs in (1, 0):
        s = hl.Solver(precision=precision, fused_small_grids=0, cuda_graphs=graphs, newton_residual_first=res_first,
                      newton_jacobian_every=every, newton_maxit=maxit, steps0=6, T=6 * 360.0)
        for _ in range(2):  # the second call replays
            out.append(s.level_batch_solve(1, xi, with_coarse=True, allow_failures=True))
        s.close()
    assert (maxit < 3) == bool((out[0][2] != 0).all())
    ok = out[0][2] == 0
    for o in out[1:]:
        assert torch.equal(o[2], out[0][2])
        assert torch.equal(o[0][ok], out[0][0][ok]) and torch.equal(o[1][ok], out[0][1][ok])
        assert o[3] == out[0][3]


def test_captured_iterations_with_retries_equal_plain_launches(hl):
    """KL inputs on which BiCGStab fails now and then: the fallback solve's own graph."""
    xi = torch.as_tensor(1.6 * inputs.kl_inputs(9300, 6), device="cuda")
    xi[:, -1].clamp_(-1.0, 1.0)
    out = []
    for graphs in (1, 0):
        s = hl.Solver(coef_model=hl.HENRY_MODEL_KL, precision=1, cuda_graphs=graphs, lin_maxit=3, steps0=4, T=4 * 360.0)
        out.append(s.level_batch_solve(1, xi, allow_failures=True))
        s.close()
    ok = out[0][2] == 0
    assert torch.equal(out[0][2], out[1][2]) and out[0][3] == out[1][3]
    assert torch.equal(out[0][0][ok], out[1][0][ok])


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("level,n,nu", [(0, 1, (2, 2)), (0, 3, (1, 2)), (1, 3, (2, 2)), (1, 2, (0, 1)), (1, 2, (1, 0)),
                                        (3, 2, (2, 1))])
def test_vertex_tail_is_bit_identical_to_separate_kernels(hl, precision, level, n, nu):
    ny, nx = 16 << level, 32 << level
    xi = torch.as_tensor(inputs.uniform_xi(9400 + level, n), device="cuda")
    b = torch.as_tensor(inputs.rng(9401 + n).standard_normal((n, ny + 1, nx + 1, 2)), device="cuda")
    z = []
    for tail in (-1, 0):
        s = hl.Solver(scheme=hl.HENRY_SCHEME_VERTEX, precision=precision, mg_tail_cells=tail, nu1=nu[0], nu2=nu[1])
        z.append(s.precondition(level, xi, _wedge(n, ny + 1, nx + 1, 0.0), _wedge(n, ny + 1, nx + 1, 0.02), b))
        s.close()
    assert bool(torch.isfinite(z[0]).all()) and torch.equal(z[0], z[1])


@pytest.mark.parametrize("res_first,every,maxit", [(2, 1, 30), (-1, 2, 30), (3, 2, 30), (2, 1, 1)])
def test_vertex_captured_iterations_equal_plain_launches(hl, res_first, every, maxit):
    xi = torch.as_tensor(inputs.uniform_xi(9500, 4), device="cuda")
    out = []
    for graphs in (1, 0):
        s = hl.Solver(scheme=hl.HENRY_SCHEME_VERTEX, cuda_graphs=graphs, newton_residual_first=res_first,
                      newton_jacobian_every=every, newton_maxit=maxit, steps0=4, T=4 * 360.0)
        out.append(s.level_batch_solve(0, xi, allow_failures=True))
        s.close()
    ok = out[0][2] == 0
    assert (maxit == 1) == bool((~ok).all())
    assert torch.equal(out[0][2], out[1][2]) and torch.equal(out[0][0][ok], out[1][0][ok]) and out[0][3] == out[1][3]


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("nu", [(2, 2), (1, 1), (3, 1), (0, 2), (2, 0)])
def test_fused_level0_solver_with_other_sweep_counts(hl, precision, nu):
    """The one-CTA-per-sample solver's V-cycle and matvec (red cells only where
    a black half-sweep ends the cycle) with the sweep counts that change their
    phases: the multi-kernel path solves to the same Newton tolerance."""
    xi = torch.as_tensor(inputs.uniform_xi(9400, 3), device="cuda")
    q = []
    for fused in (2, 0):
        s = hl.Solver(precision=precision, fused_small_grids=fused, nu1=nu[0], nu2=nu[1], steps0=6, T=6 * 360.0)
        qf, _, st, _ = s.level_batch_solve(0, xi)
        assert int(st.abs().sum()) == 0
        q.append(qf)
        s.close()
    assert torch.allclose(q[0], q[1], rtol=1e-9, atol=1e-14)


def test_concurrent_levels_build_their_graphs_over_and_over(hl):
    """Rounds of changing sizes: every level thread builds, replays and (past
    the cache's bound) drops graphs while the others do the same."""
    s = hl.Solver(steps0=2, T=720.0, max_level=2)
    h = hl.Solver(steps0=2, T=720.0, max_level=2, cuda_graphs=0)
    for k in range(60):
        levels = [0] * (3 + k % 19) + [1] * (2 + k % 17) + [2] * (1 + k % 18)
        xi = torch.as_tensor(inputs.uniform_xi(9500 + k, len(levels)), device="cuda")
        levels = torch.tensor(levels, dtype=torch.int32)
        qf, qc, st, _ = s.batch_solve_mixed(levels, xi, with_coarse=True)
        assert int(st.abs().sum()) == 0
        if k % 20 == 19:
            rf, rc, _, _ = h.batch_solve_mixed(levels, xi, with_coarse=True)
            assert torch.equal(qf, rf) and torch.equal(qc.nan_to_num(), rc.nan_to_num())
    s.close()
    h.close()
