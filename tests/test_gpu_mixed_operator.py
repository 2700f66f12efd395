"""The mixed mode's Jacobian blocks: FP32 values of the FP64 ones."""
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


@pytest.mark.parametrize("level,tile", [(0, 1), (0, 0), (1, 1), (4, 1)])
def test_diffusive_derivatives_take_three_roundings(hl, level, tile):
    """Pressure that depends on y alone: no flux crosses an east or west face,
    and the derivative of its salt flux is -phi Dm rho of the neighbour.  In
    FP32 that is phi Dm rounded, rho rounded and their product rounded: three
    roundings of 2^-24 (fixed beforehand; 2^-44 for their products)."""
    ny, nx, n = 16 << level, 32 << level, 4 if level == 4 else 64
    gen = inputs.rng(7600 + level)
    y = ((torch.arange(ny, dtype=torch.float64, device="cuda") + 0.5) / ny)[None, :, None]
    c = 0.9 + 0.1 * torch.as_tensor(gen.random((n, ny, nx)), device="cuda")
    x = torch.stack([(10000.0 * (1.0 - y)).expand(n, ny, nx), c], dim=-1).contiguous()
    xi = torch.as_tensor(inputs.uniform_xi(7601 + level, n), device="cuda")
    J = []
    for precision in (0, 1):
        s = hl.Solver(precision=precision, tile_assembly=tile)
        J.append(s.assemble(level, xi, x, x)[1])
        s.close()
    off = (J[1] / J[0] - 1.0).abs()
    assert float(off[:, :, :-1, 2, 1, 1].max()) <= 3.0 * 2.0 ** -24 + 2.0 ** -44  # east: rho of the right cell
    assert float(off[:, :, 1:, 1, 1, 1].max()) <= 3.0 * 2.0 ** -24 + 2.0 ** -44   # west: of the left one
