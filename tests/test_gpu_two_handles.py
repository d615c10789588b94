"""Two handles, or two networks, of different sizes alive at once: what the smaller one sets up
(the shared-memory limits of the kernels are the process's, not the handle's) does not take
anything from the larger one's next call, which gives its first call's bits."""
import pytest

import oracle
from synth.configs import small

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from gpu_helpers import gpu_solver  # noqa: E402

LARGE = {"b256": dict(n=(32, 16, 16), edges=([16, 16], [16], [16])),
         "b60": dict(n=(24, 20, 12), edges=([12, 12], [10, 10], [6, 6]), patch=((2, 2),) * 3),
         "b144": dict(n=(24, 24, 12), edges=([12, 12], [12, 12], [12]), patch=((4, 4),) * 3)}


@pytest.mark.parametrize("precision", ["fp32_ir", "fp64"])
@pytest.mark.parametrize("name", list(LARGE))
def test_a_smaller_handle_between_two_solves(name, precision):
    runs = []
    for kw in (LARGE[name], dict(n=(10, 9, 18), edges=([5, 5], [9], [9, 9])), dict()):
        w = small(sigma=1.0, lam=3.0, **kw)
        prob = oracle.from_workload(w)
        s = gpu_solver(w, precision, ir_tol=1e-12)
        args = torch.from_numpy(prob.K).cuda(), torch.from_numpy(prob.f).cuda()
        runs.append((s, args, [t.clone() for t in s.solve(*args)[:3]]))
    for s, args, first in runs:
        for a, b in zip(s.solve(*args)[:3], first):
            assert torch.equal(a, b)


def test_a_smaller_network_between_two_predictions():
    from paper_2103_08513_gb300.learned import WarmStartNet
    gen = torch.Generator(device="cuda").manual_seed(3)
    runs = []
    for shape in ((7, 10, 10), (2, 3, 3)):          # the first one's planes do not fit the fused pass
        net = WarmStartNet(*shape, hidden=32, layers=3, batch=4)
        x = torch.randn((4, 4, *shape), device="cuda", generator=gen)
        runs.append((net, x, net.predict(x).clone()))
    for net, x, first in runs:
        assert torch.equal(net.predict(x), first)
