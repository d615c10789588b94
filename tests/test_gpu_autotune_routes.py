"""The autotuner where the streaming solve takes some or all of the subdomains: no variant is
picked by the noise of timing one kernel twelve times, and in a model in waves, whose first
waves hold the largest blocks, the variants are timed where they are used."""
import pytest

import oracle
from synth.configs import small

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from gpu_helpers import rel_l2  # noqa: E402


def _tuned(w, **kw):
    from paper_2103_08513_gb300 import MRCM
    prob = oracle.from_workload(w)
    s = MRCM(w.n, w.edges, w.patch, precision="fp32_ir", ir_max_sweeps=8, ir_tol=1e-13, **kw)
    K, f = torch.from_numpy(prob.K).cuda(), torch.from_numpy(prob.f).cuda()
    s.factor_local(K)
    picked = s.autotune(f)
    p, u, X, _ = s.solve(K, f)
    assert rel_l2(X.cpu().numpy(), oracle.solve_mrcm(prob).X) < 1e-8
    t = s.tuning_times()
    return s, picked, t["first_solve"], t["sweeps"]


def test_blocks_of_the_streaming_solve_alone_are_timed_once(tmp_path):
    w = small(n=(24, 18, 20), edges=([12, 12], [9, 9], [10, 10]), sigma=1.0, lam=3.0)        # b = 90
    cache = tmp_path / "tune.txt"
    s, picked, first, sweeps = _tuned(w, tune_cache=str(cache))
    assert picked == (0, 0) and cache.read_text().split()[1:3] == ["0", "0"]
    assert first[0] > 0 and sweeps[0] > 0 and set(first[1:]) == {-1.0} and set(sweeps[1:]) == {-1.0}


def test_waves_are_tuned_where_a_block_takes_a_variant():
    w = small(n=(20, 24, 16), edges=([10, 4, 6], [12, 12], [10, 6]), patch=((3, 3),) * 3, sigma=1.0, lam=3.0)
    s, picked, first, sweeps = _tuned(w, wave_bytes=400 << 10)
    assert s.sizes["n_waves"] > 1
    assert min(first) > 0 and min(sweeps) > 0
