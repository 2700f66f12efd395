"""More batch sizes than a group keeps captured iterations for: two rounds of
them, the second one rebuilding what was given up, against plain launches."""
import pytest
import torch

from paper_2302_07804_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scheme,level", [(0, 0), (1, 0)])
def test_more_sizes_than_graphs(scheme, level):
    from paper_2302_07804_gb300 import henry as hl
    xi = torch.as_tensor(inputs.uniform_xi(7900, 261), device="cuda")
    q = []
    for graphs in (0, 1):
        s = hl.Solver(scheme=scheme, steps0=1, T=360.0, cuda_graphs=graphs)
        if not graphs:
            q.append(s.level_batch_solve(level, xi)[0])
        else:
            s.level_batch_solve(level, xi)  # the largest first: the workspace then stays
            for _ in range(2):
                for n in range(1, 262):
                    qf, _, st, _ = s.level_batch_solve(level, xi[:n].contiguous())
                    assert int(st.abs().sum()) == 0 and torch.equal(qf, q[0][:n]), n
        s.close()
