"""Local solves at the edges of the rules that choose a route on the GPU: FP64 products of few
columns and of column counts that leave a rest of 1, 2 or 3 past the tiles of four, subdomains
shared by several CTAs, models with slab blocks on both sides of 64 (two solve kernels side by
side), boxes with more side faces than the Robin table holds, and post-processing whose FP64
problems fill several chunks of slots.  Against the oracle; tolerances as for the solve (FP64
1e-10 relative L2, mixed 1e-8: backward-stable solves of systems of condition below 1e5)."""
import numpy as np
import pytest

import oracle
from oracle.postprocess import postprocess_mean
from synth.configs import BETA_ALPHA_H_OVER_K, small

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from gpu_helpers import rel_l2, run_gpu  # noqa: E402

# FP64: right-hand sides m = 2 nI + 1 = 3, 5, 9, 7 and more, slab blocks of 1 to 60 cells
FEW = {
    "m3_b1": dict(n=(24, 1, 1), edges=([12, 12], [1], [1])),
    "m3_b6": dict(n=(16, 3, 2), edges=([8, 8], [3], [2])),
    "m5_b16": dict(n=(15, 4, 4), edges=([5, 5, 5], [4], [4])),
    "m7_b35": dict(n=(14, 14, 5), edges=([7, 7], [7, 7], [5]), patch=((0, 0), (4, 0), (0, 0))),
    "m9_b60": dict(n=(20, 12, 5), edges=([10, 10], [12], [5]), patch=((6, 3), (0, 0), (0, 0))),
    "m27_b25": dict(n=(15, 15, 10), edges=([5, 5, 5], [5, 5, 5], [5, 5]), patch=((3, 3), (3, 3), (3, 3))),
}


@pytest.mark.parametrize("name", list(FEW))
def test_fp64_products_of_few_columns(name):
    w = small(**FEW[name])
    prob = oracle.from_workload(w)
    r = oracle.solve_mrcm(prob)
    s, p, u, X, mres, code, st = run_gpu(w, prob.K, prob.f, "fp64")
    assert code == 0, st
    assert rel_l2(p, r.p) < 1e-10 and rel_l2(u.ravel(), r.u.ravel()) < 1e-10


@pytest.mark.parametrize("name,edges", [("few", ([12, 12], [12, 8], [8, 4])), ("one_big", ([12, 6], [9], [8])),
                                        ("thin", ([12, 12, 1], [12, 1], [8]))])
def test_blocks_on_both_sides_of_64(name, edges):
    w = small(n=tuple(sum(e) for e in edges), edges=edges, sigma=1.5, lam=4.0)
    prob = oracle.from_workload(w)
    r = oracle.solve_mrcm(prob)
    s, p, u, X, mres, code, st = run_gpu(w, prob.K, prob.f, "fp32_ir", ir_max_sweeps=8, ir_tol=1e-12)
    assert st["unconverged"] == 0
    assert rel_l2(p, r.p) < 1e-8 and rel_l2(u.ravel(), r.u.ravel()) < 1e-8


@pytest.mark.parametrize("mode", ["const", "HK"])
@pytest.mark.parametrize("nz", [384, 385, 900])
def test_boxes_around_the_robin_table(mode, nz):
    """Boxes of 2 x 2 x (nz - 1) cells have 8 + 8 (nz - 1) side faces; the table holds 3072."""
    kw = dict(beta_mode=BETA_ALPHA_H_OVER_K, alpha=0.5) if mode == "HK" else {}
    w = small(n=(4, 2, nz), edges=([2, 2], [2], [nz - 1, 1]), sigma=1.0, lam=3.0, **kw)
    prob = oracle.from_workload(w)
    r = oracle.solve_mrcm(prob)
    s, p, u, X, mres, code, st = run_gpu(w, prob.K, prob.f, "fp64")
    assert code == 0, st
    assert rel_l2(p, r.p) < 1e-9 and rel_l2(u.ravel(), r.u.ravel()) < 1e-9   # 4 nz cells in a column: condition ~ nz^2


@pytest.mark.parametrize("wave_kb", [0, 300])
def test_postprocess_slots_in_chunks(wave_kb):
    from paper_2103_08513_gb300 import MRCM
    w = small(n=(24, 24, 8), edges=([6] * 4, [6] * 4, [4, 4]), patch=((3, 2), (3, 2), (3, 3)), sigma=2.5, lam=6.0)
    prob = oracle.from_workload(w)
    r = oracle.solve_mrcm(prob)
    ref = postprocess_mean(prob, r.u)
    s = MRCM(w.n, w.edges, w.patch, precision="fp32_ir", ir_max_sweeps=8, ir_tol=1e-13, wave_bytes=wave_kb << 10)
    p, u, X, mres = s.solve(torch.from_numpy(prob.K).cuda(), torch.from_numpy(prob.f).cuda())
    up, _ = s.postprocess_velocity(u.clone())
    torch.cuda.synchronize()
    assert rel_l2(up.cpu().numpy().ravel(), ref.ravel()) < 1e-8
