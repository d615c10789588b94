"""The local solve with fragment-order factors and tensor-core products (slab
blocks above 64, mixed precision) against the oracle's local solve: blocks at,
one above and one below a multiple of its 16 x 16 tiles, of the 8 x 8 factor
tiles (odd counts pad a half tile) and of the factor's CTA sizes, from the
smallest to the largest block; one column group and several (more than 16
right-hand sides), one to eight output tiles a warp; subdomains shared by several
CTAs (few of them) and not; a handle that mixes these subdomains with small ones.

Tolerance 1e-8 relative L2, the mixed bar of the other parity tests."""
import numpy as np
import pytest

import oracle
from oracle.mrcm import local_problem, solve_local
from oracle.problem import build_bases
from synth.configs import small

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

WHOLE = ((0, 0),) * 3
# (subdomain edges x, y, z), patch
CASES = [((5, 13, 13), WHOLE), ((8, 9, 10), WHOLE), ((8, 10, 11), WHOLE), ((9, 9, 10), WHOLE), ((8, 12, 9), WHOLE),
         ((10, 10, 10), ((5, 5),) * 3), ((11, 11, 11), ((4, 4),) * 3), ((8, 14, 14), ((3, 4),) * 3), ((8, 16, 16), WHOLE),
         ((3, 29, 43), WHOLE), ((8, 17, 18), WHOLE), ((12, 12, 13), ((6, 6),) * 3), ((12, 15, 16), WHOLE),
         ((14, 15, 16), WHOLE), ((15, 16, 17), WHOLE), ((16, 16, 16), ((8, 8),) * 3)]


@pytest.mark.parametrize("case", CASES)
def test_mixed_columns_match_the_oracle(case):
    from paper_2103_08513_gb300 import MRCM
    (ex, ey, ez), patch = case
    w = small(n=(2 * ex, ey, ez), edges=([ex, ex], [ey], [ez]), patch=patch, sigma=1.5, lam=3.0, beta_const=0.6,
              h=(0.5, 1.0, 2.0))
    prob = oracle.from_workload(w)
    _, sub_bases, face_basis = build_bases(prob)
    s = MRCM(w.n, w.edges, w.patch, h=w.h, beta_const=w.beta_const, precision="fp32_ir", ir_max_sweeps=8, ir_tol=1e-12)
    s.factor_local(torch.from_numpy(prob.K).cuda())
    s.solve_mbf(torch.from_numpy(prob.f).cuda())
    torch.cuda.synchronize()
    st = s.read_status()[1]
    assert st["not_spd"] == 0 and st["unconverged"] == 0 and s.read_fallback() == (0, 0)
    for l in range(2):
        want = solve_local(local_problem(prob, l, sub_bases, face_basis))
        got = s.mbf_block(l, want.shape[1], want.shape[0])
        assert np.linalg.norm(got - want.T) <= 1e-8 * np.linalg.norm(want)


def test_mixed_block_sizes_in_one_handle():
    """Small and large slab blocks in one decomposition, whole solve against the oracle."""
    from paper_2103_08513_gb300 import MRCM
    w = small(n=(24, 27, 18), edges=([12, 4, 8], [12, 12, 3], [12, 6]), patch=((4, 5),) * 3, sigma=1.5, lam=4.0)
    prob = oracle.from_workload(w)
    r = oracle.solve_mrcm(prob)
    s = MRCM(w.n, w.edges, w.patch, precision="fp32_ir", ir_max_sweeps=8, ir_tol=1e-13)
    p, u, X, _ = s.solve(torch.from_numpy(prob.K).cuda(), torch.from_numpy(prob.f).cuda())
    torch.cuda.synchronize()
    for got, want in ((p, r.p), (u, r.u), (X, r.X)):
        got = got.cpu().numpy().ravel()
        assert np.linalg.norm(got - np.ravel(want)) <= 1e-8 * np.linalg.norm(want)
