"""Workloads of the MRCM library, as a user's program calls them.

``listed()`` are the cases that are timed; ``draw(rng)`` gives more of the same
ranges; ``prepare`` makes what a program has in hand before the call (inputs on
the GPU, the handle with its workspace, network weights), ``run`` is one pass
through the public entry points, ``work`` the bytes and operations that a pass
cannot do without and ``exact`` the same outputs in plain FP64 numpy / torch.

A case is a dict of plain values.  ``kind`` is

* ``solve``: the whole pressure solve (`MRCM.solve`, or `MRCM.solve_host` with
  page-locked host buffers), K and f in, p, u and X out;
* ``impes``: the two-phase loop (`MRCM.impes`): pressure solve, velocity
  post-processing and transport steps, the saturation out;
* ``learned``: the pressure solve whose basis functions come from warm-started
  conjugate gradients, network prediction included;
* ``predict`` / ``gradient``: the warm-start network on its own (inference of
  every sample of a solve; the gradient of one training batch);
* ``box``: the allocation-free local solve of one box.

Subdomain edges are ``"10x10x5"`` (the last one along an axis truncated to fit)
or ``"random 8,12,16"`` (drawn per axis from the list, the last truncated).
The mass residual that a solve also writes is left out of the outputs: it is
the rounding error of a sum that vanishes exactly.  Mixed-precision cases stop
a column at 1e-10 (a tenth of the benchmark's stop) so that two correct
programs agree to well below 1e-9.
"""
from __future__ import annotations

import ctypes as C
import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_2103_08513_gb300 import MRCM, _lib
from paper_2103_08513_gb300.learned import WarmStartNet


def _solve(name, n, edges, patch, **kw):
    case = dict({"name": name} if name else {}, kind="solve", nx=n[0], ny=n[1], nz=n[2], edges=edges, edge_seed=0, patch=patch,
                precision="fp32_ir", sweeps=6, tol=1e-10, field="lognormal", sigma=2.0, lam=8.0, kz=0.1,
                wells="five", beta="const", alpha=1.0, walls="noflow", graph=False, tune=False, host=False,
                wave_mb=0, refine=-1)
    case.update(kw)
    return case


def listed():
    return [
        # one local problem, solved by code that may not allocate (a plug-in, a real-time loop): the smallest call
        dict(name="box_10x10x5", kind="box", nx=10, ny=10, nz=5, sides="robin", sigma=2.0),
        # the small reference configuration in FP64 with the default settings: a sector model, latency-bound
        _solve("solve_40x40x8_fp64", (40, 40, 8), "10x10x4", "5x2", precision="fp64", wells="corner", refine=0),
        # a small model of awkward sizes: truncated subdomains, odd slab blocks, beta = alpha H / K, fixed
        # pressure on two walls, called step by step with the default interface refinement
        _solve("solve_45x38x27_ragged_mixed", (45, 38, 27), "10x9x7", "4x3", beta="HK", walls="dirichlet_x",
               refine=0),
        # the benchmark's reservoir model (SPE10 shape, layered) in a time loop: tuned handle, replayed graph
        _solve("solve_60x220x85_mixed_graph", (60, 220, 85), "10x10x5", "5x5", field="layered", sigma=3.0,
               graph=True, tune=True),
        # the same model called from a host program: K, f from and p, u, X to page-locked host buffers
        _solve("solve_60x220x85_mixed_host", (60, 220, 85), "10x10x5", "5x5", field="layered", sigma=3.0,
               graph=True, tune=True, host=True),
        # the same model in plain FP64 (the form a user checks the mixed one against)
        _solve("solve_60x220x85_fp64", (60, 220, 85), "10x10x5", "5x5", field="layered", sigma=3.0,
               precision="fp64"),
        # uneven subdomains (slab blocks of 64 to 256 cells), whole-face interface spaces
        _solve("solve_256x256x128_uneven_mixed", (256, 256, 128), "random 8,12,16", "whole", sigma=2.5),
        # a large model whose block factors are bounded to 2 GB at a time (four waves), high contrast
        _solve("solve_256x512x128_waves_mixed", (256, 512, 128), "16x16x8", "whole", sigma=3.0, kz=0.05, sweeps=8,
               wave_mb=2048),
        # two-phase simulation: one pressure solve, velocity post-processing, ten transport steps
        dict(_solve("impes_60x220x85_mixed", (60, 220, 85), "10x10x5", "5x5", field="layered", sigma=3.0),
             kind="impes", skip=10, steps=10),
        # the learned form on its own workload: sample gathering, prediction, CG inside FP64 refinement
        dict(_solve("learned_40x40x10", (40, 40, 10), "10x10x5", "5x2", precision="learned_pcg", wells="corner",
                    tol=1e-11), kind="learned", hidden=32, layers=4, batch=256),
        # network inference on every sample of such a solve
        dict(name="predict_896", kind="predict", depth=5, height=10, width=10, hidden=32, layers=4, batch=256, count=896),
        # one training batch: loss and gradient (the optimiser's update is a cheap pass over the same array)
        dict(name="gradient_256", kind="gradient", depth=5, height=10, width=10, hidden=32, layers=4, batch=256,
             count=256, weighted=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "solve", "solve", "impes", "learned", "predict", "gradient", "box"])
    if kind == "box":
        return dict(kind="box", nx=rng.randint(3, 11), ny=rng.randint(2, 11), nz=rng.randint(1, 16),
                    sides=rng.choice(["robin", "mixed"]), sigma=rng.choice([1.0, 2.0, 3.0]))
    if kind in ("predict", "gradient"):
        return dict(kind=kind, depth=rng.randint(3, 8), height=rng.randint(4, 10), width=rng.randint(4, 10),
                    hidden=rng.choice([8, 16, 32, 32]), layers=rng.randint(3, 5), batch=256,
                    count=_log_int(rng, 8, 1200) if kind == "predict" else _log_int(rng, 8, 256),
                    weighted=rng.random() < 0.5)
    if kind == "learned":
        e = rng.choice(["10x10x5", "8x8x6", "9x7x5"])
        return dict(_solve("", (rng.randint(18, 44), rng.randint(18, 44), rng.randint(8, 14)), e, "5x2",
                           precision="learned_pcg", wells="corner", tol=1e-11, sigma=rng.choice([1.0, 1.5, 2.0])),
                    kind="learned", hidden=rng.choice([16, 32]), layers=4, batch=256)
    if kind == "impes":
        nx, ny = rng.randint(50, 70), rng.randint(90, 200)
        c = _solve("", (nx, ny, rng.randint(40, 80)), rng.choice(["10x10x5", "9x10x6", "12x8x5"]), "5x5",
                   field="layered", sigma=rng.choice([2.0, 3.0]))
        steps = rng.randint(4, 10)
        return dict(c, kind="impes", skip=steps, steps=steps)
    # a whole solve: cell counts over three decades, aspect ratios and remainders at random
    coarse = rng.random() < 0.35
    cells = _log_int(rng, 8e3, 4e6 if coarse else 8e5)
    nz = max(4, min(128, int(round((cells / 12.0) ** (1.0 / 3.0) * rng.uniform(0.6, 1.4)))))
    nx = max(8, int(round(math.sqrt(cells / nz) * rng.uniform(0.5, 1.5))))
    ny = max(8, int(round(cells / (nz * nx))))
    graph = rng.random() < 0.5
    if coarse:
        edges = rng.choice(["16x16x8", "random 8,12,16", "12x12x8", "13x11x9"])
        patch = "whole"
    else:
        edges = rng.choice(["10x10x5", "10x10x4", "8x8x8", "9x10x6", "11x7x5", "random 6,8,10"])
        patch = rng.choice(["5x5", "whole", "5x2" if edges.startswith("10x10") else "4x4"])
    fp64 = cells < 3e5 and rng.random() < 0.35
    return _solve("", (nx, ny, nz), edges, patch, edge_seed=rng.randint(0, 99), precision="fp64" if fp64 else "fp32_ir",
                  sweeps=8, field=rng.choice(["lognormal", "layered"]), sigma=rng.choice([1.0, 2.0, 2.5]),
                  kz=rng.choice([0.02, 0.1, 0.3]), wells=rng.choice(["five", "corner"]),
                  beta=rng.choice(["const", "const", "HK"]), walls=rng.choice(["noflow", "noflow", "dirichlet_x"]),
                  graph=graph, host=graph and rng.random() < 0.3, refine=rng.choice([-1, 0]))


# ---------------------------------------------------------------- inputs
_side = {}


def _stream():
    """The program's own stream (graph replay needs one that is not the default)."""
    d = torch.cuda.current_device()
    if d not in _side:
        _side[d] = torch.cuda.Stream(d)
    return _side[d]


def _gen(seed, salt):
    return torch.Generator(device="cuda").manual_seed(1000003 * int(seed) + salt)


def _gauss(shape, sigma, lam, gen):
    """Gaussian field with covariance sigma^2 exp(-r / lam) on the periodic grid (circulant square root)."""
    r2 = torch.zeros((), dtype=torch.float64, device="cuda")
    for a, n in enumerate(shape):
        d = torch.arange(n, dtype=torch.float64, device="cuda")
        d = torch.minimum(d, n - d) ** 2
        r2 = r2 + d.reshape([-1 if b == a else 1 for b in range(len(shape))])
    eig = torch.fft.rfftn(sigma * sigma * torch.exp(-r2.sqrt() / lam)).real.clamp_(min=0.0)
    w = torch.randn(shape, dtype=torch.float64, device="cuda", generator=gen)
    return torch.fft.irfftn(eig.sqrt_() * torch.fft.rfftn(w), s=shape)


def _permeability(c, seed):
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    gen = _gen(seed, 1)
    K = torch.empty((3, nz, ny, nx), dtype=torch.float64, device="cuda")
    if c["field"] == "layered":
        par = np.random.RandomState(seed % (1 << 31))
        for k in range(nz):
            kx = _gauss((ny, nx), c["sigma"], float(par.uniform(4.0, 20.0)), gen).exp()
            K[0, k] = kx
            K[2, k] = float(10.0 ** par.uniform(-3.0, -1.0)) * kx
    else:
        kx = _gauss((nz, ny, nx), c["sigma"], c["lam"], gen).exp()
        K[0] = kx
        K[2] = c["kz"] * kx
    K[1] = K[0]
    return K


def _wells(c):
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    f = torch.zeros((nz, ny, nx), dtype=torch.float64)
    if c["wells"] == "corner":
        f[:, 0, 0] += 1.0 / nz
        f[:, ny - 1, nx - 1] -= 1.0 / nz
    else:
        f[:, ny // 2, nx // 2] += 1.0 / nz
        for j, i in ((0, 0), (0, nx - 1), (ny - 1, 0), (ny - 1, nx - 1)):
            f[:, j, i] -= 0.25 / nz
    return f.cuda()


def _edges(c):
    n = (c["nx"], c["ny"], c["nz"])
    if c["edges"].startswith("random"):
        rng = np.random.Generator(np.random.PCG64(c["edge_seed"]))
        choices = [int(v) for v in c["edges"].split()[1].split(",")]
        out = []
        for m in n:
            e = []
            while sum(e) < m:
                e.append(min(int(rng.choice(choices)), m - sum(e)))
            out.append(e)
        return out
    return [[e] * (m // e) + ([m % e] if m % e else []) for m, e in zip(n, (int(v) for v in c["edges"].split("x")))]


def _patch(c):
    p = (0, 0) if c["patch"] == "whole" else tuple(int(v) for v in c["patch"].split("x"))
    return (p, p, p)


def _handle(c, allocate=True):
    dirichlet = c["walls"] == "dirichlet_x"
    return MRCM((c["nx"], c["ny"], c["nz"]), _edges(c), _patch(c), beta_mode=1 if c["beta"] == "HK" else 0,
                alpha=c["alpha"], bc_type=((1, 1) if dirichlet else (0, 0), (0, 0), (0, 0)),
                bc_value=((1.0, 0.0) if dirichlet else (0.0, 0.0), (0.0, 0.0), (0.0, 0.0)), precision=c["precision"],
                ir_max_sweeps=c["sweeps"], ir_tol=c["tol"], wave_bytes=c["wave_mb"] << 20,
                interface_refine=c["refine"], allocate=allocate)


def _channels(c):
    return [4] + [c["hidden"]] * (c["layers"] - 1), [c["hidden"]] * (c["layers"] - 1) + [1]


def _weights(c, seed):
    """He-normal weights (output layer a tenth of that), small biases: the flat master vector, FP32."""
    gen = torch.Generator().manual_seed(7919 * int(seed) + 3)
    parts = []
    for l, (ci, co) in enumerate(zip(*_channels(c))):
        s = math.sqrt(2.0 / (27.0 * ci)) * (0.1 if l + 1 == c["layers"] else 1.0)
        parts += [torch.randn(co * ci * 27, generator=gen) * s, torch.randn(co, generator=gen) * 0.02]
    parts[-1] -= 1.5
    return torch.cat(parts)


def _net(c, seed, shape):
    net = WarmStartNet(*shape, hidden=c["hidden"], layers=c["layers"], batch=c["batch"])
    net.master.copy_(_weights(c, seed))
    net.sync_weights()
    return net


def _samples(c, seed):
    """Network inputs like those of `mrcm_net_samples`: log K / 4 (x and z), one basis' faces, all Robin faces."""
    D, H, W, n = c["depth"], c["height"], c["width"], c["count"]
    gen = _gen(seed, 5)
    x = torch.zeros((n, 4, D, H, W), device="cuda")
    g = F.avg_pool3d(torch.randn((n, 1, D, H, W), device="cuda", generator=gen), 3, 1, 1)[:, 0] * 6.0
    x[:, 0] = 0.25 * g
    x[:, 1] = 0.25 * (g - 2.3)
    x[:, 2, :, : (H + 1) // 2, W - 1] = 1.0
    x[:, 3, :, :, 0] = x[:, 3, :, :, W - 1] = x[:, 3, :, 0] = x[:, 3, :, H - 1] = 1.0
    x[:, 3, 0] = x[:, 3, D - 1] = 1.0
    t = torch.rand((n, 1, D, H, W), device="cuda", generator=gen) ** 3
    w = x[:, 3:4] * torch.rand((n, 1, D, H, W), device="cuda", generator=gen)
    return x, t, w


def _box_inputs(c, seed):
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    gen = _gen(seed, 9)
    K = (c["sigma"] * torch.randn((3, nz, ny, nx), dtype=torch.float64, device="cuda", generator=gen)).exp()
    f = torch.randn((nz, ny, nx), dtype=torch.float64, device="cuda", generator=gen)
    nf = 2 * (ny * nz + nx * nz + nx * ny)
    g = torch.randn(nf, dtype=torch.float64, device="cuda", generator=gen)
    beta = 0.5 + torch.rand(nf, dtype=torch.float64, device="cuda", generator=gen)
    side = [1] * 6 if c["sides"] == "robin" else [0, 1, 1, 2, 1, 0]
    return K, f, g, beta, side


def prepare(case, seed):
    c = case
    if c["kind"] == "box":
        K, f, g, beta, side = _box_inputs(c, seed)
        out = (torch.empty_like(f), torch.empty_like(g), torch.empty(1, dtype=torch.int32, device="cuda"))
        return dict(c=c, lib=_lib.load(), K=K, f=f, g=g, beta=beta, out=out,
                    box=(C.c_int * 3)(c["nx"], c["ny"], c["nz"]), h=(C.c_double * 3)(1.0, 1.0, 1.0),
                    side=(C.c_int * 6)(*side))
    if c["kind"] in ("predict", "gradient"):
        x, t, w = _samples(c, seed)
        return dict(c=c, net=_net(c, seed, (c["depth"], c["height"], c["width"])), x=x, t=t,
                    w=w if c.get("weighted") else None)
    K, f = _permeability(c, seed), _wells(c)
    s = _handle(c)
    st = dict(c=c, s=s, K=K, f=f, out=s.outputs())
    if c["kind"] == "learned":
        st["net"] = _net(c, seed, tuple(e[0] for e in reversed(_edges(c))))
    if c["kind"] == "impes":
        st["S0"] = torch.zeros_like(f)
        st["S"] = torch.zeros_like(f)
    if c["tune"]:
        s.factor_local(K)
        s.autotune(f)
    if c["host"]:
        st["out"] = tuple(torch.empty_like(t, device="cpu").pin_memory() for t in st["out"])
        st["K"], st["f"] = K.cpu().pin_memory(), f.cpu().pin_memory()
    torch.cuda.synchronize()
    return st


# ---------------------------------------------------------------- one pass
def run(state):
    c = state["c"]
    kind = c["kind"]
    if kind == "box":
        p, q, flag = state["out"]
        ptr = [C.c_void_p(t.data_ptr()) for t in (state["K"], state["f"], state["g"], state["beta"], p, q, flag)]
        rc = state["lib"].mrcm_box_solve_noalloc(state["box"], state["h"], state["side"], *ptr,
                                                 C.c_void_p(torch.cuda.current_stream().cuda_stream))
        if rc:
            raise RuntimeError("mrcm_box_solve_noalloc: %d" % rc)
        return {"p": p, "q": q, "not_spd": flag}
    if kind == "predict":
        return state["net"].predict(state["x"])
    if kind == "gradient":
        grad, loss = state["net"].gradient(state["x"], state["t"], weight=state["w"])
        return {"grad": grad, "loss": loss}
    s, K, f = state["s"], state["K"], state["f"]
    if kind == "impes":
        S = state["S"]
        S.copy_(state["S0"])
        t = s.impes(K, f, S, C_skip=c["skip"], n_steps=c["steps"])
        return {"S": S, "t": t}
    if kind == "learned":
        X, p, u, mres = state["out"]
        s.factor_local(K)
        x, _ = state["net"].samples(s, targets=False)
        pred = state["net"].predict(x)
        s.solve_mbf_learned(f, net=state["net"], pred=pred)
        s.assemble_interface()
        s.solve_interface(X)
        s.reconstruct(X, p, u, mres)
        return {"p": p, "u": u, "X": X}
    stream = _stream() if c["graph"] else None
    X, p, u, mres = state["out"]
    if c["host"]:
        s.solve_host(K, f, X, p, u, mres, stream=stream, graph=c["graph"])
    else:
        s.solve(K, f, out=state["out"], stream=stream, graph=c["graph"])
    return {"p": p, "u": u, "X": X}


# ---------------------------------------------------------------- what a pass cannot do without
def work(case):
    c = case
    if c["kind"] == "box":
        dims = sorted((c["nx"], c["ny"], c["nz"]))
        n, b = dims[0] * dims[1] * dims[2], dims[0] * dims[1]
        nf = 2 * (c["nx"] * c["ny"] + c["ny"] * c["nz"] + c["nx"] * c["nz"])
        return {"bytes": 8.0 * (5 * n + 3 * nf), "flops": float(n) * b * b + 4.0 * n * b}
    if c["kind"] in ("predict", "gradient"):
        vox = c["depth"] * c["height"] * c["width"] * c["count"]
        mac = sum(27 * ci * co for ci, co in zip(*_channels(c)))
        if c["kind"] == "predict":
            return {"bytes": 4.0 * 5 * vox, "flops": 2.0 * mac * vox}
        # backward: the weights' gradient of every layer, the data's of all but the first
        return {"bytes": 4.0 * 6 * vox, "flops": 2.0 * vox * (3 * mac - 27 * 4 * c["hidden"])}
    # banded Cholesky of every local matrix, one solve of every column with it, the interface LDL^T
    z = _handle(c, allocate=False).sizes
    n = c["nx"] * c["ny"] * c["nz"]
    flops = z["local_factor_flops"] + z["local_solve_flops"] + z["ldl_flops"]
    if c["kind"] == "impes":
        return {"bytes": 8.0 * 6 * n, "flops": flops + z["local_factor_flops"] + 60.0 * n * c["steps"]}
    return {"bytes": 8.0 * (11 * n + 2 * z["n_basis"]), "flops": flops}


# ---------------------------------------------------------------- the same in plain FP64
def _tpfa(K):
    """Dense matrix of the interior faces of one box (unit cells): K (3, nz, ny, nx)."""
    nz, ny, nx = K.shape[1:]
    idx = np.arange(nx * ny * nz).reshape(nz, ny, nx)
    A = np.zeros((idx.size, idx.size))
    trans = []
    for a in range(3):
        ax = 2 - a
        lo, hi = [slice(None)] * 3, [slice(None)] * 3
        lo[ax], hi[ax] = slice(0, -1), slice(1, None)
        k1, k2 = K[a][tuple(lo)], K[a][tuple(hi)]
        T = 2.0 * k1 * k2 / (k1 + k2)
        i, j, t = idx[tuple(lo)].ravel(), idx[tuple(hi)].ravel(), T.ravel()
        np.add.at(A, (i, i), t)
        np.add.at(A, (j, j), t)
        A[i, j] -= t
        A[j, i] -= t
        trans.append((lo, hi, T))
    return idx, A, trans


def _exact_box(c, seed):
    K, f, g, beta, side = _box_inputs(c, seed)
    K, f, g, beta = (t.cpu().numpy() for t in (K, f, g, beta))
    idx, A, _ = _tpfa(K)
    rhs = f.reshape(-1).copy()
    faces, off = [], 0
    for a in range(3):
        for hi in (0, 1):
            sl = [slice(None)] * 3
            sl[2 - a] = -1 if hi else 0
            cell, kn = idx[tuple(sl)].ravel(), K[a][tuple(sl)].ravel()
            sel = slice(off, off + cell.size)
            off += cell.size
            sd = side[2 * a + hi]
            T = 1.0 / (0.5 / kn + beta[sel]) if sd == 1 else 2.0 * kn if sd == 2 else np.zeros(cell.size)
            A[cell, cell] += T
            rhs[cell] += T * g[sel]
            faces.append((cell, T, sel))
    p = np.linalg.solve(A, rhs)
    q = np.zeros_like(g)
    for cell, T, sel in faces:
        q[sel] = T * (p[cell] - g[sel])
    return {"p": p.reshape(f.shape), "q": q, "not_spd": None}


def _exact_net(c, seed):
    x, t, w = (v.double() for v in _samples(c, seed))
    master = _weights(c, seed).to(x.device)
    params, off = [], 0
    for ci, co in zip(*_channels(c)):
        k = co * ci * 27
        params.append(master[off:off + k].bfloat16().double().reshape(co, ci, 3, 3, 3).requires_grad_())
        params.append(master[off + k:off + k + co].double().requires_grad_())
        off += k + co

    def net(v):
        for l in range(c["layers"]):
            v = F.conv3d(v, params[2 * l], params[2 * l + 1], padding=1)
            v = torch.sigmoid(v) if l + 1 == c["layers"] else F.leaky_relu(v, 0.01)
        return v

    if c["kind"] == "predict":
        with torch.no_grad():
            return net(x)
    d = (net(x) - t) ** 2
    loss = ((1.0 + w) * d if c.get("weighted") else d).mean()
    loss.backward()
    return {"grad": torch.cat([v.grad.reshape(-1) for v in params]), "loss": loss.detach().reshape(1)}


def _exact_solve(c, seed):
    """The method step by step (Robin problems per subdomain, interface system, reconstruction), dense FP64."""
    n = (c["nx"], c["ny"], c["nz"])
    edges, patch = _edges(c), _patch(c)
    sub_cells = max(edges[0]) * max(edges[1]) * max(edges[2])
    nsub = len(edges[0]) * len(edges[1]) * len(edges[2])
    if nsub * float(sub_cells) ** 3 > 1.5e11:
        return None
    K, f = _permeability(c, seed).cpu().numpy(), _wells(c).cpu().numpy()
    dirichlet = c["walls"] == "dirichlet_x"
    starts = [np.concatenate([[0], np.cumsum(e)]) for e in edges]
    N = [len(e) for e in edges]
    sid = lambda i: i[0] + N[0] * (i[1] + N[1] * i[2])  # noqa: E731
    # interface basis functions: by normal axis, lower subdomain, patch (second tangential axis slow)
    subs = [(i, j, k) for k in range(N[2]) for j in range(N[1]) for i in range(N[0])]
    first, nv = {}, 0
    for a in range(3):
        t1, t2 = [x for x in range(3) if x != a]
        for ijk in subs:
            if ijk[a] + 1 < N[a]:
                e1, e2 = edges[t1][ijk[t1]], edges[t2][ijk[t2]]
                q1, q2 = patch[a][0] or e1, patch[a][1] or e2
                m1, m2 = -(-e1 // q1), -(-e2 // q2)
                first[(a, sid(ijk))] = (nv, q1, q2, m1)
                nv += m1 * m2
    if 2 * nv > 5000:
        return None
    A = np.zeros((2 * nv, 2 * nv))
    b = np.zeros(2 * nv)
    keep = []
    for ijk in subs:
        lo = [int(starts[a][ijk[a]]) for a in range(3)]
        sz = [edges[a][ijk[a]] for a in range(3)]
        box = (slice(lo[2], lo[2] + sz[2]), slice(lo[1], lo[1] + sz[1]), slice(lo[0], lo[0] + sz[0]))
        Kb, fb = K[(slice(None),) + box], f[box]
        idx, M, trans = _tpfa(Kb)
        part = fb.reshape(-1).copy()
        robin, walls = [], []
        for a in range(3):
            t1, t2 = [x for x in range(3) if x != a]
            for hi in (0, 1):
                sl = [slice(None)] * 3
                sl[2 - a] = -1 if hi else 0
                cell, kn = idx[tuple(sl)].ravel(), Kb[a][tuple(sl)].ravel()
                if (ijk[a] + 1 == N[a]) if hi else (ijk[a] == 0):
                    if a == 0 and dirichlet:
                        T, gv = 2.0 * kn, (0.0 if hi else 1.0)
                        M[cell, cell] += T
                        part[cell] += T * gv
                        walls.append((hi, sl, cell, T, gv))
                    continue
                lower = list(ijk)
                lower[a] -= 0 if hi else 1
                base, q1, q2, m1 = first[(a, sid(lower))]
                c2, c1 = np.meshgrid(np.arange(sz[t2]), np.arange(sz[t1]), indexing="ij")
                basis = (base + c1 // q1 + m1 * (c2 // q2)).ravel()
                beta = c["alpha"] * sz[a] / kn if c["beta"] == "HK" else np.ones_like(kn)
                T = 1.0 / (0.5 / kn + beta)
                M[cell, cell] += T
                robin.append((cell, basis, T, beta, np.full(cell.size, 1.0 if hi else -1.0), a, hi, sl))
        cell, basis, T, beta, s = (np.concatenate([r[i] for r in robin]) for i in range(5))
        own = np.unique(basis)
        col = np.searchsorted(own, basis)
        m = own.size
        B = np.zeros((idx.size, 2 * m + 1))
        np.add.at(B, (cell, col), T)
        np.add.at(B, (cell, m + col), -beta * s * T)
        B[:, 2 * m] = part
        Y = np.linalg.solve(M, B)
        G = np.zeros((cell.size, 2 * m + 1))
        G[np.arange(cell.size), col] = 1.0
        G[np.arange(cell.size), m + col] = -beta * s
        q = T[:, None] * (Y[cell] - G)
        rows = np.zeros((2 * m, 2 * m + 1))
        np.add.at(rows, col, q)
        np.add.at(rows, m + col, (beta * s)[:, None] * q)
        np.add.at(rows, (m + col, m + col), -beta)
        dofs = np.concatenate([own, nv + own])
        A[np.ix_(dofs, dofs)] += rows[:, :-1]
        b[dofs] -= rows[:, -1]
        keep.append((box, idx, trans, robin, walls, dofs, Y))
    if not dirichlet:
        A[0] = 0.0
        A[0, 0] = 1.0
        b[0] = 0.0
    X = np.linalg.solve(A, b)
    X += np.linalg.solve(A, b - A @ X)
    p = np.zeros(f.shape)
    u = np.zeros((6,) + f.shape)
    for box, idx, trans, robin, walls, dofs, Y in keep:
        v = Y @ np.concatenate([X[dofs], [1.0]])
        pb = v[idx]
        p[box] = pb
        ub = np.zeros((6,) + pb.shape)
        for a, (lo, hi, T) in enumerate(trans):
            flux = T * (pb[tuple(lo)] - pb[tuple(hi)])
            ub[2 * a + 1][tuple(lo)] = flux
            ub[2 * a][tuple(hi)] = flux
        for cell, basis, T, beta, s, a, hi, sl in robin:
            flux = s * T * (v[cell] - (X[basis] - beta * s * X[nv + basis]))
            ub[2 * a + hi][tuple(sl)] = flux.reshape(pb[tuple(sl)].shape)
        for hi, sl, cell, T, gv in walls:
            flux = (1.0 if hi else -1.0) * T * (v[cell] - gv)
            ub[hi][tuple(sl)] = flux.reshape(pb[tuple(sl)].shape)
        u[(slice(None),) + box] = ub
    if not dirichlet:
        p -= p.mean()
    return {"p": p, "u": u, "X": X}


def exact(case, seed):
    if case["kind"] == "box":
        return _exact_box(case, seed)
    if case["kind"] in ("predict", "gradient"):
        return _exact_net(case, seed)
    if case["kind"] == "impes":
        return None        # a whole two-phase run of a million cells: minutes in plain FP64
    return _exact_solve(case, seed)
