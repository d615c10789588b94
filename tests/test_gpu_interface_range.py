"""The interface's right-hand side goes through the fronts with the emulated FP64 update, whose
integer slices have no NaN or infinity: what is not finite has to reach every unknown all the
same, as it does in FP64 (the top of the elimination tree couples them all)."""
import numpy as np
import pytest

import oracle
from synth.configs import small

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from gpu_helpers import gpu_solver  # noqa: E402

BC = {"noflow": {}, "dirichlet": dict(bc_type=((1, 1), (0, 0), (0, 0)), bc_value=((0.0, 0.0),) * 3)}


def _model():
    # the parity test's big_fronts: fronts of up to 144 eliminated dofs, most of their steps emulated
    return small(n=(36, 36, 12), edges=([6] * 6, [6] * 6, [4, 4, 4]), patch=((3, 2), (3, 2), (3, 3)), sigma=1.5, lam=4.0)


def _solve(w, K, f, precision="fp64", **kw):
    s = gpu_solver(w, precision, **kw)
    p, u, X, _ = s.solve(torch.from_numpy(K).cuda(), torch.from_numpy(f).cuda())
    torch.cuda.synchronize()
    return X.cpu().numpy(), p.cpu().numpy()


@pytest.mark.parametrize("value", [np.nan, np.inf])
@pytest.mark.parametrize("refine", [-1, 0])
@pytest.mark.parametrize("walls", list(BC))
def test_a_source_that_is_not_finite_leaves_no_finite_unknown(walls, refine, value):
    w = _model()
    prob = oracle.from_workload(w, **BC[walls])
    f = prob.f.copy()
    f[2, 3, 4] = value
    X, p = _solve(w, prob.K, f, interface_refine=refine, **BC[walls])
    assert not np.isfinite(X).any() and not np.isfinite(p).any()
