"""Post-processing whose FP64 problems fill one chunk of slots, several with a last one that is
partly filled, and many of two: the same bits whatever the chunks.  The field is layered, six
decades wide, which half of the tied Neumann blocks' FP32 factors do not survive; the counts are
asserted.  (No comparison with the oracle here: the stop on the backward error, 1e-13, leaves
1e-13 times the blocks' condition in the velocity, which for such a field is no small number;
test_gpu_postprocess.py compares at ordinary contrast.)"""
import numpy as np
import pytest

import oracle
from synth.configs import small

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _field(nx, ny, nz):
    rng = np.random.default_rng(1)
    K = np.empty((3, nz, ny, nx))
    K[0] = 10.0 ** (rng.uniform(-3, 3, (nz, 1, 1)) + rng.uniform(-1, 1, (nz, ny, nx)))
    K[1] = K[0]
    K[2] = K[0] * 10.0 ** rng.uniform(-3, -1, (nz, 1, 1))
    return K


def test_slots_in_one_chunk_or_several():
    from paper_2103_08513_gb300 import MRCM
    w = small(n=(24, 24, 8), edges=([6] * 4, [6] * 4, [4, 4]), patch=((3, 2), (3, 2), (3, 3)), sigma=1.0, lam=6.0)
    prob = oracle.from_workload(w)
    prob = oracle.from_workload(w, K=_field(24, 24, 8), f=prob.f)
    per_sub = 6 * 24 * 24 * 4                    # bytes of one subdomain's FP32 factors (6 slabs of 24 cells)
    first = None
    for wave_kb in (0, 200, 60):
        s = MRCM(w.n, w.edges, w.patch, precision="fp32_ir", ir_max_sweeps=8, ir_tol=1e-13, wave_bytes=wave_kb << 10)
        p, u, X, mres = s.solve(torch.from_numpy(prob.K).cuda(), torch.from_numpy(prob.f).cuda())
        up, _ = s.postprocess_velocity(u.clone())
        torch.cuda.synchronize()
        count, lost = s.read_fallback()
        slots = ((wave_kb << 10) // per_sub if wave_kb else 32) // 2        # of a chunk: twice the bytes in FP64
        assert lost == 0 and s.read_status()[1]["unconverged"] == 0
        assert count <= slots if not wave_kb else count > slots and count % slots != 0
        if first is None:
            first = up
            assert torch.isfinite(up).all()
        assert torch.equal(up, first)
