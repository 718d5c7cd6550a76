"""Timed workloads of the library, as a program that uses it runs them.

Kinds of work:
  solve    one lattice: load a medium, advance it, read K_app and the velocity
           field (``Solver``) -- the library's main path
  batch    a sweep of uneven media advanced together (``Batch``)
  predict  the learned warm start's network on a medium's features
           (``surrogate.UNet.forward_tc``)
  conv     one 3x3 layer of that network (``glbm_nn_tc_conv``)
  train    one training step of that network on the tensor cores
  em       the Gaussian-mixture fit of pore radii (``em_gmm1d``)

Fields and gradients come back in the type that their precision is: FP32 for
FP32 storage, BF16 for 16-bit storage and for the BF16 network.
"""

import ctypes
import math

import numpy as np
import torch
import torch.nn.functional as F

import paper_1601_00704_gb300 as glbm
from paper_1601_00704_gb300 import surrogate
from paper_1601_00704_gb300 import train_surrogate as T

TAU = 1.0
NU = (TAU - 0.5) / 3.0
G = 1e-6


# -- the cases ---------------------------------------------------------------

def solve(nx, ny, storage, n, check, tol=0.0, walls=True, F_eps=0.0, stream=True):
    return {"kind": "solve", "nx": nx, "ny": ny, "storage": storage, "n": n, "check": check, "tol": tol,
            "walls": walls, "F_eps": F_eps, "stream": stream}


def listed():
    return [
        # a small sample run with the convergence test on, as in the README (the 128 x 128 parity workload): latency and launches
        dict(solve(128, 128, "f32", 500, 100, tol=1e-10), name="solve_128_f32"),
        # an image-sized sample of odd width, periodic, with Forchheimer drag, on the default stream (one node per thread)
        dict(solve(333, 517, "f32", 200, 100, walls=False, F_eps=0.5, stream=False), name="solve_333x517_forch"),
        # a 512-node-wide sample in BF16 storage
        dict(solve(512, 384, "bf16", 500, 100), name="solve_512x384_bf16"),
        # the 8 um shale matrix at 1024 nodes: fits the L2 cache
        dict(solve(1024, 1024, "f32", 500, 100, tol=1e-10), name="solve_1024_f32"),
        # the warm-start study's lattice in FP16 storage, whose scale is checked every chunk
        dict(solve(2048, 2048, "f16", 300, 100, tol=1e-10), name="solve_2048_f16"),
        # the benchmark's lattice, FP32 and BF16 storage
        dict(solve(4096, 4096, "f32", 200, 100), name="solve_4096_f32"),
        dict(solve(4096, 4096, "bf16", 200, 100), name="solve_4096_bf16"),
        # a pressure / Langmuir sweep over uneven media, sides of 64 to 1024 as in the batched benchmark
        {"kind": "batch", "count": 24, "lo": 64, "hi": 1024, "storage": "f32", "n": 200, "check": 100, "name": "batch_24_f32"},
        # warm start of a 2048 x 2048 medium with the committed network
        {"kind": "predict", "h": 2048, "w": 2048, "name": "predict_2048"},
        # its 128-channel layer with a skip input (d2a of a 2048 x 2048 medium)
        {"kind": "conv", "n": 1, "h": 512, "w": 512, "c0": 128, "c1": 128, "cout": 128, "name": "conv_512_256to128"},
        # a training step of the committed architecture on the recipe's batch of 256 x 256 media
        {"kind": "train", "n": 8, "h": 256, "w": 256, "name": "train_8x256"},
        # pore radii of an OM/IOM image split into two components
        {"kind": "em", "m": 1000000, "k": 2, "iters": 50, "name": "em_1m_2"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "solve", "batch", "predict", "conv", "train", "em"])
    if kind == "solve":
        nx = _log_int(rng, 64, 4096)
        ny = min(4096, max(48, int(nx * rng.uniform(0.5, 2.0))))
        if rng.random() < 0.75:
            nx = nx // 4 * 4
        most = (2 if nx % 4 == 0 else 1) * 10 ** 9 // (nx * ny)
        n = max(40, min(most, rng.randrange(100, 600)))
        return solve(nx, ny, rng.choice(["f32", "f32", "bf16", "f16"]), n, rng.choice([20, 50, 64, 100, 101, 250]),
                     tol=rng.choice([0.0, 1e-10]), walls=rng.random() < 0.7, F_eps=rng.choice([0.0, 0.0, 0.0, 0.5, -1.0]),
                     stream=rng.random() < 0.75)
    if kind == "batch":
        return {"kind": "batch", "count": rng.randrange(3, 25), "lo": 64, "hi": rng.choice([256, 512, 1024]),
                "storage": rng.choice(["f32", "f32", "bf16"]), "n": rng.randrange(50, 201), "check": rng.choice([25, 50, 100])}
    if kind == "predict":
        return {"kind": "predict", "h": 32 * _log_int(rng, 2, 64), "w": 32 * _log_int(rng, 2, 64)}
    if kind == "conv":
        side = _log_int(rng, 16, 1024)
        c0, cout = rng.choice([32, 64, 128]), rng.choice([32, 64, 128, 128])
        return {"kind": "conv", "n": rng.choice([1, 1, 2, 4]) if side < 512 else 1, "h": side,
                "w": max(16, int(side * rng.uniform(0.5, 2.0))) if side < 512 else side,
                "c0": c0, "c1": rng.choice([0, 0, cout]), "cout": cout}
    if kind == "train":
        return {"kind": "train", "n": rng.randrange(1, 9), "h": 32 * rng.randrange(2, 9), "w": 32 * rng.randrange(2, 9)}
    return {"kind": "em", "m": _log_int(rng, 1000, 2000000), "k": rng.randrange(1, 5), "iters": rng.randrange(5, 51)}


# -- inputs ------------------------------------------------------------------

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _organic(ny, nx, gen, frac=0.2, ell=8.0):
    """OM mask: the largest values of a Gaussian random field of correlation length ell."""
    noise = torch.randn((ny, nx), generator=gen, device="cuda")
    kx = 2 * math.pi * torch.fft.rfftfreq(nx, device="cuda")
    ky = 2 * math.pi * torch.fft.fftfreq(ny, device="cuda")
    filt = torch.exp(-(ky[:, None] ** 2 + kx[None, :] ** 2) * ell ** 2 / 4)
    field = torch.fft.irfft2(torch.fft.rfft2(noise) * filt, s=(ny, nx))
    cut = field.flatten().sort().values[int((1 - frac) * nx * ny)]
    return field >= cut


def _medium(ny, nx, gen, shale=False):
    """eps and K per node (FP64): the two-phase medium of the benchmark, or the OM/IOM medium of the network's recipe."""
    om = _organic(ny, nx, gen)
    if shale:
        z = torch.randn((ny, nx), generator=gen, device="cuda", dtype=torch.float64)
        r = torch.where(om, 5e-9, 20e-9).double() * torch.exp(0.5 * z)
        eps = torch.where(om, 0.04, 0.02).double()
        K = eps * (2 * r) ** 2 / (32 * T.TORT) / T.DX ** 2 * 4 + 1e-5
        return eps, K
    u = torch.rand((ny, nx), generator=gen, device="cuda", dtype=torch.float64)
    eps = torch.where(om, 0.15, 0.10).double()
    K = torch.where(om, 10 ** (math.log10(5e-4) + u), 10 ** (-4 + u))
    return eps, K


def _sides(case, seed):
    rng = np.random.default_rng(seed)
    return [(4 * int(a), 4 * int(b)) for a, b in rng.integers(case["lo"] // 4, case["hi"] // 4 + 1, size=(case["count"], 2))]


def _batch_shapes(case):
    return _sides(case, 12345)


def _net(seed):
    """The committed architecture with random weights of that scale."""
    return surrogate.UNet(base=32, levels=6, max_ch=128, seed=int(seed) % (1 << 31))


def _conv_inputs(case, seed):
    gen = _gen(seed)
    n, h, w, c0, c1, co = (case[k] for k in ("n", "h", "w", "c0", "c1", "cout"))

    def act(c):
        return torch.randn((n, h, w, c), generator=gen, device="cuda").relu_().to(torch.bfloat16)
    x0, x1 = act(c0), act(c1) if c1 else None
    wt = (torch.randn((co, c0 + c1, 3, 3), generator=gen, device="cuda") * math.sqrt(2.0 / (9 * (c0 + c1)))).contiguous()
    bias = 0.1 * torch.randn(co, generator=gen, device="cuda")
    return x0, x1, wt, bias


def _train_inputs(case, seed):
    gen = _gen(seed)
    shape = (case["n"], 3, case["h"], case["w"])
    return torch.randn(shape, generator=gen, device="cuda"), torch.randn(shape, generator=gen, device="cuda")


def _em_inputs(case, seed):
    gen = _gen(seed)
    k = case["k"]
    which = torch.randint(0, k, (case["m"],), generator=gen, device="cuda")
    mu = torch.tensor([5.0 + 6.0 * j for j in range(k)], dtype=torch.float64, device="cuda")  # nm, overlapping
    x = mu[which] + (1.5 + 0.8 * which) * torch.randn(case["m"], generator=gen, device="cuda", dtype=torch.float64)
    return x, [1.0 / k] * k, [3.0 + 7.0 * j for j in range(k)], [9.0] * k


class State:
    pass


def prepare(case, seed):
    s = State()
    s.case, kind = case, case["kind"]
    if kind == "solve":
        nx, ny = case["nx"], case["ny"]
        s.eps, s.K = _medium(ny, nx, _gen(seed))
        s.stream = torch.cuda.Stream() if case["stream"] else torch.cuda.default_stream()
        s.u = [torch.empty((ny, nx), dtype=torch.float64, device="cuda") for _ in range(2)]
        s.out = [torch.empty((ny, nx), dtype=torch.float32 if case["storage"] == "f32" else torch.bfloat16, device="cuda")
                 for _ in range(2)]
        torch.cuda.synchronize()
        s.solver = glbm.Solver(nx, ny, tau=TAU, storage=case["storage"], walls=case["walls"],
                               stream=s.stream if case["stream"] else None)
        s.solver.set_force(G)
    elif kind == "batch":
        gen = _gen(seed)
        s.batch = glbm.Batch(_batch_shapes(case), tau=TAU, storage=case["storage"])
        for i, (ny, nx) in enumerate(s.batch.shapes):
            eps, K = _medium(ny, nx, gen)
            torch.cuda.synchronize()
            s.batch.set_medium(i, eps, K)
        s.batch.set_force(G)
    elif kind == "predict":
        s.net = _net(seed)
        eps, K = _medium(case["h"], case["w"], _gen(seed), shale=True)
        s.x = torch.stack([(eps - 0.05) / 0.05, (K.log10() + 2) / 2, torch.zeros_like(eps)]).float()[None].contiguous()
    elif kind == "conv":
        s.x0, s.x1, w, s.bias = _conv_inputs(case, seed)
        n, h, wd, co, ci = case["n"], case["h"], case["w"], case["cout"], case["c0"] + case["c1"]
        s.lib = glbm.load()
        s.w = torch.empty((9, co, ci), dtype=torch.bfloat16, device="cuda")
        rc = s.lib.glbm_nn_tc_pack_weights(_p(w), co, ci, 3, co, ci, _p(s.w), _stream())
        torch.cuda.synchronize()
        if rc:
            raise RuntimeError("pack_weights: %d" % rc)
        s.y = torch.empty((n, h, wd, co), dtype=torch.bfloat16, device="cuda")
        s.err = torch.zeros(1, dtype=torch.int32, device="cuda")
    elif kind == "train":
        s.net = _net(seed)
        s.x, s.t = _train_inputs(case, seed)
        s.start = s.net.params.clone()
    else:
        s.x, s.phi, s.mu, s.var = _em_inputs(case, seed)
    return s


def _p(t):
    return ctypes.c_void_p(t.data_ptr()) if t is not None else None


def _stream():
    return ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)


# -- one pass ----------------------------------------------------------------

def run(s):
    case, kind = s.case, s.case["kind"]
    if kind == "solve":
        v = s.solver
        v.set_medium(s.eps, s.K, F_eps=case["F_eps"])
        v.step(case["n"], tol=case["tol"], check_every=case["check"])
        kxx = v.permeability()
        v.velocity(*s.u)
        with torch.cuda.stream(s.stream):
            for o, u in zip(s.out, s.u):
                o.copy_(u)
        return {"kxx": kxx, "ux": s.out[0], "uy": s.out[1]}
    if kind == "batch":
        b = s.batch
        b.reset()
        b.step(case["n"], check_every=case["check"])
        r = b.results()
        # a sweep keeps K and U of every medium; the fields are looked at for one
        ux = b.fields(0)[1]
        return {"kxx": r["kxx"].astype(np.float32), "ux": r["mean_u"][:, 0].astype(np.float32), "steps": r["steps"],
                "field": ux.astype(np.float32)}
    if kind == "predict":
        return s.net.forward_tc(s.x).to(torch.bfloat16)
    if kind == "conv":
        n, h, w, co = case["n"], case["h"], case["w"], case["cout"]
        rc = s.lib.glbm_nn_tc_conv(_p(s.x0), case["c0"], _p(s.x1), case["c1"], n, h, w, 3, _p(s.w), _p(s.bias), co,
                                   _p(s.y), co, 1, 0, 0, _p(s.err), _stream())
        if rc:
            raise RuntimeError("tc_conv: %d" % rc)
        return s.y
    if kind == "train":
        net = s.net
        net.params.copy_(s.start)  # every pass is the first step from these weights
        net.m.zero_(), net.v.zero_()
        net.t = 0
        net.invalidate_tc()
        pred = net.forward(s.x, tc=True)
        loss, g = net.loss(pred, s.t, T.CHANNEL_WEIGHT)
        net.backward(g, tc=True)
        net.adam_step(1e-3)
        # every convolution takes BF16 operands: so precise are the prediction and the gradients
        return {"loss": loss.float(), "pred": pred.to(torch.bfloat16), "grads": net.grads.to(torch.bfloat16)}
    phi, mu, var, it, ll = glbm.em_gmm1d(s.x, s.phi, s.mu, s.var, max_iter=case["iters"], tol=1e-8)
    return {"phi": phi, "mu": mu, "var": var, "it": it, "ll": np.array([ll])}


# -- what a pass cannot do without -------------------------------------------

NODE_FLOPS = 180  # Eqs. 30-37 per node and time step


def _unet_flops(h, w, n):
    return surrogate.UNet.flops(_Shape, h, w, n)


class _Shape:
    """Layer table of the committed architecture (as surrogate.UNet's), for its operation count."""
    levels = 6
    ch = [32, 64, 128, 128, 128, 128]
    specs = ([("e0a", 3, 32, 3), ("e0b", 32, 32, 3), ("e1a", 32, 64, 3), ("e1b", 64, 64, 3), ("e2a", 64, 128, 3)]
             + [(f"e{l}{x}", 128, 128, 3) for l in range(2, 6) for x in "ab" if (l, x) != (2, "a")]
             + [(f"d{l}{x}", 256 if x == "a" else 128, 128, 3) for l in (4, 3, 2) for x in "ab"]
             + [("d1a", 192, 64, 3), ("d1b", 64, 64, 3), ("d0a", 96, 32, 3), ("d0b", 32, 32, 3), ("head", 32, 3, 1)])


def work(case):
    kind = case["kind"]
    if kind == "solve":
        nodes = case["nx"] * case["ny"]
        return {"bytes": nodes * (16 + 2 * (4 if case["storage"] == "f32" else 2)), "flops": NODE_FLOPS * nodes * case["n"]}
    if kind == "batch":
        nodes = sum(a * b for a, b in _batch_shapes(case))
        return {"bytes": 8 * nodes, "flops": NODE_FLOPS * nodes * case["n"]}
    if kind == "predict":
        return {"bytes": case["h"] * case["w"] * (12 + 6), "flops": _unet_flops(case["h"], case["w"], 1)}
    if kind == "conv":
        px, ci = case["n"] * case["h"] * case["w"], case["c0"] + case["c1"]
        return {"bytes": 2 * px * (ci + case["cout"]) + 18 * ci * case["cout"], "flops": 18 * px * ci * case["cout"]}
    if kind == "train":
        px = case["n"] * case["h"] * case["w"]
        return {"bytes": px * (12 + 12 + 6) + 7 * 4 * 2684995, "flops": 3 * _unet_flops(case["h"], case["w"], case["n"])}
    return {"bytes": 8 * case["m"], "flops": 60 * case["m"] * case["k"] * case["iters"]}


# -- the same in 64 bits -----------------------------------------------------

EX, EY = (0, 1, 0, -1, 0, 1, -1, -1, 1), (0, 0, 1, 0, -1, 1, 1, -1, -1)
OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)


def _lattice(eps, K, n, walls, F_eps):
    """n steps of Eqs. 27-37 from rest, deviations g = f - w: (ux, uy) of the last step's collision."""
    w = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4
    alpha = eps * NU / K
    beta = 0.0 if F_eps == 0 else eps * (F_eps if F_eps > 0 else 1.75 / (150 * eps ** 3).sqrt()) / K.sqrt()
    g = [torch.zeros_like(eps) for _ in range(9)]
    c0 = 0.5 + 0.25 * alpha
    om, A = 1 / TAU, 1 - 0.5 / TAU
    ux = uy = None
    for _ in range(n):
        s = []
        for i in range(9):
            t = torch.roll(g[i], (EY[i], EX[i]), (0, 1)) if i else g[0]
            if walls and EY[i] == 1:
                t[0] = g[OPP[i]][0]
            elif walls and EY[i] == -1:
                t[-1] = g[OPP[i]][-1]
            s.append(t)
        d = sum(s[1:], s[0])
        rho = 1 + d
        vx = (s[1] - s[3] + s[5] - s[6] - s[7] + s[8]) / rho + 0.5 * eps * G
        vy = (s[2] - s[4] + s[5] + s[6] - s[7] - s[8]) / rho
        if F_eps == 0:
            den = 2 * c0
        else:
            den = c0 + (c0 * c0 + 0.5 * beta * (vx * vx + vy * vy).sqrt()).sqrt()
        ux, uy = vx / den, vy / den
        drag = alpha + beta * (ux * ux + uy * uy).sqrt() if F_eps != 0 else alpha
        fx, fy = eps * G - drag * ux, -drag * uy
        uu, uf = (ux * ux + uy * uy) / eps, (ux * fx + uy * fy) / eps
        for i in range(9):
            eu, ef = EX[i] * ux + EY[i] * uy, EX[i] * fx + EY[i] * fy
            eq = w[i] * (d + rho * (3 * eu + 4.5 * eu * eu / eps - 1.5 * uu))
            s[i] = s[i] + om * (eq - s[i]) + w[i] * A * rho * (3 * ef + 9 * eu * ef / eps - 3 * uf)
        g = s
    return ux, uy


def _unet64(net, x, params):
    def conv(t, name, relu=True):
        _, ci, co, k = next(sp for sp in net.specs if sp[0] == name)
        a, b = net.offsets[name]
        t = F.conv2d(t, params[a:b].view(co, ci, k, k), params[b:b + co], padding=k // 2)
        return t.relu() if relu else t
    skips, t = [], x
    for l in range(net.levels):
        t = conv(conv(t, f"e{l}a"), f"e{l}b")
        if l < net.levels - 1:
            skips.append(t)
            t = F.avg_pool2d(t, 2)
    for l in range(net.levels - 2, -1, -1):
        t = torch.cat([t.repeat_interleave(2, 2).repeat_interleave(2, 3), skips[l]], 1)
        t = conv(conv(t, f"d{l}a"), f"d{l}b")
    return conv(t, "head", relu=False)


def exact(case, seed):
    kind = case["kind"]
    if kind == "solve":
        eps, K = _medium(case["ny"], case["nx"], _gen(seed))
        ux, uy = _lattice(eps, K, case["n"], case["walls"], case["F_eps"])
        return {"kxx": float(NU * ux.mean() / G), "ux": ux, "uy": uy}
    if kind == "batch":
        gen, k, u, field = _gen(seed), [], [], None
        for ny, nx in _batch_shapes(case):
            eps, K = _medium(ny, nx, gen)
            ux, _ = _lattice(eps, K, case["n"], True, 0.0)
            field = ux.cpu().numpy() if field is None else field
            u.append(float(ux.mean()))
            k.append(NU * u[-1] / G)
        return {"kxx": np.array(k), "ux": np.array(u), "steps": None, "field": field}
    if kind == "predict":
        if case["h"] * case["w"] > 1 << 20:
            return None  # FP64 convolutions of that size take too long
        s = prepare(case, seed)
        with torch.no_grad():
            return _unet64(s.net, s.x.double(), s.net.params.double())
    if kind == "conv":
        if case["n"] * case["h"] * case["w"] * (case["c0"] + case["c1"]) * case["cout"] > 1 << 35:
            return None
        x0, x1, w, b = _conv_inputs(case, seed)
        x = x0 if x1 is None else torch.cat([x0, x1], 3)
        y = F.conv2d(x.double().permute(0, 3, 1, 2), w.to(torch.bfloat16).double(), b.double(), padding=1)
        return y.relu().permute(0, 2, 3, 1).contiguous()
    if kind == "train":
        net = _net(seed)
        x, t = _train_inputs(case, seed)
        p = net.params.double().requires_grad_()
        pred = _unet64(net, x.double(), p)
        cw = torch.tensor(T.CHANNEL_WEIGHT, dtype=torch.float64, device="cuda")
        loss = (cw * ((pred - t.double()) ** 2).mean((0, 2, 3))).sum()
        grads, = torch.autograd.grad(loss, p)
        return {"loss": loss.detach().reshape(1), "pred": pred.detach(), "grads": grads}
    x, phi, mu, var = _em_inputs(case, seed)
    phi, mu, var = (torch.tensor(v, dtype=torch.float64, device="cuda") for v in (phi, mu, var))
    ll = prev = torch.tensor(-math.inf, dtype=torch.float64, device="cuda")
    for _ in range(case["iters"]):
        d = x[:, None] - mu
        g = phi / (2 * math.pi * var).sqrt() * torch.exp(-0.5 * d * d / var)
        den = g.sum(1)
        ll = den.log().mean()
        r = g / den[:, None]
        tot = r.sum(0)
        mu = (r * x[:, None]).sum(0) / tot
        var = (r * (x[:, None] - mu) ** 2).sum(0) / tot
        phi = tot / x.numel()
        if abs(float(ll - prev)) < 1e-8:
            break
        prev = ll
    return {"phi": phi.cpu().numpy(), "mu": mu.cpu().numpy(), "var": var.cpu().numpy(), "it": None, "ll": np.array([float(ll)])}
