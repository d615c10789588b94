"""Interface solution on the GPU at the edges of the fronts' panels and tiles: fronts whose
eliminated and boundary dofs leave one row, one column or one beyond a full panel, the
right-hand side's row included, with and without a refinement step, against the oracle.
Tolerance: the FP64 form's 1e-10 relative L2 (backward-stable elimination of a quasi-definite
system scaled to unit diagonal, condition below 1e5)."""
import numpy as np
import pytest

import oracle
from synth.configs import small

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from gpu_helpers import gpu_solver, rel_l2  # noqa: E402

# (cells, subdomain edges, patches): eliminated dofs of the fronts 2 (one basis), 16 (one full
# pair), 30, 32, 34 (a panel and one pair), 66 (two panels and a remainder), odd patch counts
CASES = {
    "one_basis": ((8, 4, 4), ([4, 4], [4], [4]), ((0, 0),) * 3),
    "panel_minus": ((6, 15, 2), ([3, 3], [15], [2]), ((1, 2), (1, 1), (1, 1))),
    "panel_exact": ((6, 16, 2), ([3, 3], [16], [2]), ((1, 2), (1, 1), (1, 1))),
    "panel_plus": ((6, 17, 2), ([3, 3], [17], [2]), ((1, 2), (1, 1), (1, 1))),
    "two_panels_plus": ((6, 33, 2), ([3, 3], [33], [2]), ((1, 2), (1, 1), (1, 1))),
    "three_levels": ((12, 11, 10), ([4, 4, 4], [5, 6], [5, 5]), ((2, 2), (2, 3), (3, 2))),
}


@pytest.mark.parametrize("refine", [-1, 0])
@pytest.mark.parametrize("walls", ["noflow", "dirichlet"])
@pytest.mark.parametrize("name", list(CASES))
def test_interface_edges_match_oracle(name, walls, refine):
    n, edges, patch = CASES[name]
    bc = {}
    if walls == "dirichlet":
        bc = dict(bc_type=((1, 1), (0, 0), (0, 0)), bc_value=((1.0, 0.0), (0.0, 0.0), (0.0, 0.0)))
    w = small(n=n, edges=edges, patch=patch, sigma=1.0, lam=3.0)
    prob = oracle.from_workload(w, **bc)
    r = oracle.solve_mrcm(prob)
    s = gpu_solver(w, "fp64", interface_refine=refine, **bc)
    p, u, X, mres = s.solve(torch.from_numpy(prob.K).cuda(), torch.from_numpy(prob.f).cuda())
    torch.cuda.synchronize()
    code, st = s.read_status()
    assert st["interface_zero_pivots"] == 0
    assert rel_l2(p.cpu().numpy().ravel(), r.p) < 1e-10
    assert rel_l2(u.cpu().numpy().ravel(), r.u.ravel()) < 1e-10
