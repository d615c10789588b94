"""A column of the mixed local solve does not depend on the kernel that solves it: subdomains
of the same matrix whose number of right-hand sides lies on both sides of the limit of the
streaming solve (and, below it, at one, two and four tiles a thread) give the same bits in the
columns that they share.  The products are FP32 sums in the same order everywhere, so there is
no tolerance.

The shared columns are those of the one interface normal to x and the particular column; the
patches of the interface normal to y set the count.  Subdomain edges reach each factor kernel
above b = 64: 8 x 8 tiles (b 90, 128) and the triangle's four CTA sizes (144, 169, 240, 256)."""
import os
import subprocess

import numpy as np
import pytest

import oracle
from synth.configs import small

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# subdomain edges, slab block, patches normal to y (the last one past the limit)
CASES = [((9, 10, 10), 90, [(0, 0), (1, 2), (1, 1)]), ((8, 16, 16), 128, [(0, 0), (2, 4), (2, 2), (2, 1)]),
         ((12, 12, 12), 144, [(0, 0), (2, 2), (2, 1)]), ((13, 13, 13), 169, [(0, 0), (3, 2), (3, 1)]),
         ((15, 16, 16), 240, [(0, 0), (5, 2), (4, 2)]), ((16, 16, 16), 256, [(0, 0), (4, 4), (4, 2)])]


@pytest.fixture(scope="module")
def streams(tmp_path_factory):
    """big_ok(b, m): whether the streaming solve takes the subdomain."""
    d = tmp_path_factory.mktemp("rule")
    (d / "rule.cpp").write_text('#include <cstdio>\n#include <cstdlib>\n#include "mrcm_internal.h"\n'
                                'int main(int, char** v) { printf("%d", mrcm::big_ok(atoi(v[1]), atoi(v[2])) ? 1 : 0); }\n')
    exe = str(d / "rule")
    subprocess.check_call(["g++", "-std=c++17", "-I", os.path.join(ROOT, "paper_2103_08513_gb300", "csrc"), "-I",
                           os.path.join(ROOT, "include"), "-I", "/usr/local/cuda/include", str(d / "rule.cpp"), "-o", exe])
    return lambda b, m: subprocess.check_output([exe, str(b), str(m)]) == b"1"


@pytest.mark.parametrize("edge,b,patches", CASES)
def test_a_column_has_the_same_bits_on_every_route(edge, b, patches, streams):
    from paper_2103_08513_gb300 import MRCM
    ex, ey, ez = edge
    first = None
    for k, patch in enumerate(patches):
        q = [p or n for p, n in zip(patch, (ex, ez))]
        nI = 1 + -(-ex // q[0]) * -(-ez // q[1])
        m = 2 * nI + 1
        assert streams(b, m) == (k + 1 < len(patches))
        w = small(n=(2 * ex, 2 * ey, ez), edges=([ex, ex], [ey, ey], [ez]), patch=((0, 0), patch, (0, 0)), sigma=2.5, lam=6.0)
        prob = oracle.from_workload(w)
        s = MRCM(w.n, w.edges, w.patch, precision="fp32_ir", ir_max_sweeps=8, ir_tol=1e-10, fallback_cap=-1)
        s.factor_local(torch.from_numpy(prob.K).cuda())
        s.solve_mbf(torch.from_numpy(prob.f).cuda())
        torch.cuda.synchronize()
        got = [s.mbf_block(l, m, ex * ey * ez)[[0, nI, m - 1]] for l in range(4)]
        if first is None:
            first = got
            assert all(np.isfinite(x).all() and np.abs(x[:2]).max() > 0 for x in got)
        for x, y in zip(got, first):
            assert np.array_equal(x, y)


def test_both_routes_above_64_in_one_handle(streams):
    """Subdomains of 16 x 16 x 16 cells past the limit (b 256, 65 right-hand sides) beside
    16 x 9 x 16 below it (b 144, 57): the two kernels of a pass side by side, against the
    oracle (1e-8 relative L2, the mixed bar of the parity tests)."""
    from gpu_helpers import rel_l2, run_gpu
    assert not streams(256, 65) and streams(144, 57)
    w = small(n=(32, 25, 16), edges=([16, 16], [16, 9], [16]), patch=((4, 4),) * 3, sigma=1.5, lam=4.0)
    prob = oracle.from_workload(w)
    r = oracle.solve_mrcm(prob)
    s, p, u, X, mres, code, st = run_gpu(w, prob.K, prob.f, "fp32_ir", ir_max_sweeps=8, ir_tol=1e-13)
    assert s.sizes["max_rhs"] == 65 and st["not_spd"] == 0 and st["unconverged"] == 0
    assert rel_l2(p, r.p) < 1e-8 and rel_l2(u.ravel(), r.u.ravel()) < 1e-8 and rel_l2(X, r.X) < 1e-8


def test_post_processing_has_the_same_bits_on_either_route(streams):
    """The one column of the post-processing's FP32 pass: subdomains of 6 x 11 x 12 cells below the
    limit and, with 96 patches, past it, on the same multiscale velocity."""
    from paper_2103_08513_gb300 import MRCM
    assert streams(66, 5) and not streams(66, 193)
    first = None
    for patch, m in ((((0, 0), (0, 0), (0, 0)), 5), (((3, 2), (1, 1), (0, 0)), 193)):
        w = small(n=(12, 22, 12), edges=([6, 6], [11, 11], [12]), patch=patch, sigma=2.5, lam=6.0)
        prob = oracle.from_workload(w)
        s = MRCM(w.n, w.edges, w.patch, precision="fp32_ir", ir_max_sweeps=8, ir_tol=1e-12)
        assert s.sizes["max_rhs"] == m and s.sizes["max_block"] == 66
        p, u, X, _ = s.solve(torch.from_numpy(prob.K).cuda(), torch.from_numpy(prob.f).cuda())
        if first is None:
            given = u.clone()
        up, _ = s.postprocess_velocity(given.clone())
        torch.cuda.synchronize()
        first = up if first is None else first
        assert torch.isfinite(up).all() and torch.equal(up, first)
