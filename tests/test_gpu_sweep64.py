"""FP64 block inversion on register tiles (the batched factor and the
allocation-free box solve) at the edges of its tile and CTA sizes, against the
oracle's local solve: slab blocks b one below, at and one above a whole number
of 4 x 4 tiles and of the CTA sizes (52, 64, 96, 128), blocks spread over a
cluster (144, 176, 182, 240, 256), the smallest blocks, and an odd and an even
number of slabs (the box solve eliminates from both ends; it takes b <= 128).

Tolerance 1e-10 relative L2, the FP64 bar of the other parity tests."""
import ctypes as C

import numpy as np
import pytest

import oracle
from oracle.mrcm import local_problem, solve_local
from oracle.problem import build_bases
from synth.configs import small

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# (two shorter edges, longest edge): b = product of the first two
BOXES = [((12, 12), 13), ((11, 16), 17), ((13, 14), 14), ((15, 16), 17), ((16, 16), 16), ((1, 1), 2), ((1, 3), 4), ((3, 17), 17), ((4, 13), 14), ((6, 9), 9), ((7, 9), 10), ((8, 8), 9), ((5, 13), 14),
         ((5, 19), 20), ((8, 12), 13), ((7, 14), 15), ((8, 16), 16), ((5, 5), 5), ((2, 2), 2)]


def _problem(box):
    """Two subdomains of the same box side by side (along x), Robin on the shared side."""
    (e1, e2), e3 = box
    w = small(n=(2 * e1, e2, e3), edges=([e1, e1], [e2], [e3]), patch=((0, 0),) * 3, sigma=2.0, lam=3.0,
              beta_const=0.6, h=(0.5, 1.0, 2.0))
    return w, oracle.from_workload(w)


@pytest.mark.parametrize("box", BOXES)
def test_fp64_factor_matches_the_oracle(box):
    from paper_2103_08513_gb300 import MRCM
    w, prob = _problem(box)
    _, sub_bases, face_basis = build_bases(prob)
    s = MRCM(w.n, w.edges, w.patch, h=w.h, beta_const=w.beta_const, precision="fp64")
    s.factor_local(torch.from_numpy(prob.K).cuda())
    s.solve_mbf(torch.from_numpy(prob.f).cuda())
    torch.cuda.synchronize()
    assert s.read_status()[1]["not_spd"] == 0
    for l in range(2):
        want = solve_local(local_problem(prob, l, sub_bases, face_basis))
        m, N = want.shape[1], want.shape[0]
        got = s.mbf_block(l, m, N)
        assert np.linalg.norm(got - want.T) <= 1e-10 * np.linalg.norm(want)


@pytest.mark.parametrize("box", [x for x in BOXES if x[0][0] * x[0][1] <= 128])
def test_box_solve_matches_the_oracle(box):
    from paper_2103_08513_gb300 import _lib
    w, prob = _problem(box)
    _, sub_bases, face_basis = build_bases(prob)
    want = solve_local(local_problem(prob, 0, sub_bases, face_basis))[:, -1]      # the particular column
    (e1, e2), e3 = box
    nf = 2 * (e1 * e2 + e1 * e3 + e2 * e3)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    K, f = dev(prob.K[:, :, :, :e1]), dev(prob.f[:, :, :e1])
    g, beta = torch.zeros(nf, dtype=torch.float64, device="cuda"), torch.full((nf,), 0.6, dtype=torch.float64, device="cuda")
    p, q = torch.empty(e1 * e2 * e3, dtype=torch.float64, device="cuda"), torch.empty_like(g)
    flag = torch.full((1,), -1, dtype=torch.int32, device="cuda")
    rc = _lib.load().mrcm_box_solve_noalloc((C.c_int * 3)(e1, e2, e3), (C.c_double * 3)(*w.h),
                                            (C.c_int * 6)(0, 1, 0, 0, 0, 0),
                                            *[C.c_void_p(t.data_ptr()) for t in (K, f, g, beta, p, q, flag)],
                                            C.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == 0
    assert int(flag.cpu()[0]) == 0
    assert np.linalg.norm(p.cpu().numpy() - want) <= 1e-10 * np.linalg.norm(want)
