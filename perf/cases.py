"""The calls whose speed matters to a user of this library, as measurable cases.

Each case is one call (or one short sequence of calls) through the public entry
points of ``paper_2404_03313_gb300``, on inputs like the paper's: piecewise
constant scenes of a few smooth spectra with Gaussian noise, salt-and-pepper and
vertical stripes.  Kinds of case:

* ``solve``   ``Solver.solve`` for a fixed budget of passes of Alg. 1, cold start
              included, under one of the step-size policies, block layouts and
              regularisation functions;
* ``resume``  the stepping interface as a long solve uses it: a problem that is
              set up stays on the GPU, each call advances it by some passes and
              reads the whole P-PDS state back, block duals included;
* ``batch``   ``Solver.solve_batched`` on several cubes of uneven size;
* ``net``     the learned warm start's network, inference on one cube;
* ``train``   its gradient on a batch of crops, the work of a training step;
* ``quality`` MPSNR, MSSIM and SAM of a restored cube against its reference.
"""
from __future__ import annotations

import math

import torch
import torch.nn.functional as F

import paper_2404_03313_gb300 as P
from paper_2404_03313_gb300 import _binding as B

NET_LAYERS = ((1, 32), (32, 32), (32, 64), (64, 64), (64, 128), (128, 128), (192, 64), (64, 64), (96, 32), (32, 32))
NET_LEVEL = (0, 0, 1, 1, 2, 2, 1, 1, 0, 0)  # pooling level each convolution runs at
REGS = {"s3ttv": B.REG_S3TTV, "sstv": B.REG_SSTV}


def _solve(name, N1, N2, N3, k, passes, exact_steps=False, stacked=False, reg="s3ttv", sigma=0.1, p_t=0.05):
    return {"name": name, "kind": "solve", "N1": N1, "N2": N2, "N3": N3, "k": k, "passes": passes,
            "exact_steps": exact_steps, "stacked": stacked, "reg": reg, "sigma": sigma, "p_t": p_t}


def listed():
    return [
        # the smallest solve in use: the parity cube, where every pass is a chain of short launches
        _solve("solve_32x32x16_k3", 32, 32, 16, 3, 100),
        # an ordinary cube with odd and ragged sides (an image crop, 61 of its bands), exact Lemma 1 steps
        _solve("solve_97x131x61_k4", 97, 131, 61, 4, 40, exact_steps=True),
        # the headline workload under the paper's printed step sizes
        _solve("solve_256x256x128_k5", 256, 256, 128, 5, 40, sigma=0.05, p_t=0.10),
        # the largest cube in use (191 bands, so padded rows); a solve to the stop rule continued after a look at
        # its state: 20 passes a call under the step sizes that let the rule fire
        {"name": "resume_304x304x191_k5", "kind": "resume", "N1": 304, "N2": 304, "N3": 191, "k": 5, "passes": 20,
         "sigma": 0.1, "p_t": 0.05},
        # the paper's own scene size and 10 x 10 blocks
        _solve("solve_100x100x198_k10", 100, 100, 198, 10, 12, exact_steps=True),
        # the stacked block matrices with the open spectral boundary
        _solve("solve_128x128x64_k5_stacked", 128, 128, 64, 5, 20, stacked=True),
        # a comparison regulariser without blocks: the elementwise kernels and the l1-ball projections alone
        _solve("solve_256x256x128_sstv", 256, 256, 128, 1, 60, reg="sstv"),
        # many cubes of uneven size at once
        {"name": "batch_12_uneven", "kind": "batch", "count": 12, "lo": 64, "hi": 160, "shapes": 1, "passes": 32},
        # the warm start's prediction for the headline cube
        {"name": "net_256x256x128", "kind": "net", "N1": 256, "N2": 256, "N3": 128},
        # one training step's gradient at the training default: four 32^3 crops
        {"name": "train_4x32x32x32", "kind": "train", "batch": 4, "N1": 32, "N2": 32, "N3": 32},
        # evaluation of a restored headline cube, with its SAM map
        {"name": "quality_256x256x128", "kind": "quality", "N1": 256, "N2": 256, "N3": 128},
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("solve", "solve", "solve", "resume", "batch", "net", "train", "quality"))
    if kind == "net":  # sides are multiples of 4
        return {"kind": kind, "N1": 4 * _logint(rng, 8, 64), "N2": 4 * _logint(rng, 8, 64),
                "N3": 4 * _logint(rng, 4, 32)}
    if kind == "train":
        return {"kind": kind, "batch": rng.randint(1, 8), "N1": 4 * rng.randint(4, 10), "N2": 4 * rng.randint(4, 10),
                "N3": 4 * rng.randint(4, 10)}
    if kind == "batch":
        return {"kind": kind, "count": rng.randint(3, 12), "lo": 48, "hi": rng.randint(80, 160),
                "shapes": rng.randint(2, 10000), "passes": rng.choice((16, 32))}
    N1, N2, N3 = _logint(rng, 24, 256), _logint(rng, 24, 256), _logint(rng, 12, 198)
    if kind == "quality":
        return {"kind": kind, "N1": N1, "N2": N2, "N3": N3}
    sigma, p_t = rng.choice((0.05, 0.1)), rng.choice((0.0, 0.05, 0.1))
    if kind == "resume":
        return {"kind": kind, "N1": N1, "N2": N2, "N3": N3, "k": rng.randint(2, 5), "passes": rng.randint(8, 20),
                "sigma": sigma, "p_t": p_t}
    if rng.random() < 0.15:
        return {key: v for key, v in _solve("", N1, N2, N3, 1, rng.randint(20, 60), reg="sstv", sigma=sigma,
                                            p_t=p_t).items() if key != "name"}
    stacked = rng.random() < 0.2
    k = rng.randint(2, 5) if stacked or rng.random() < 0.6 else rng.randint(6, 10)
    if k > 5 or stacked:  # the costlier blocks come on scenes of up to about 120 x 120 pixels
        N1, N2 = min(N1, 120), min(N2, 120)
    passes = rng.randint(8, 12) if k > 5 else rng.randint(10, 40)
    c = _solve("", N1, N2, N3, k, passes, rng.random() < 0.5, stacked, "s3ttv", sigma, p_t)
    del c["name"]
    return c


# ---------------------------------------------------------------- inputs
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _scene(N1, N2, N3, g, regions=None, endmembers=5):
    """Clean cube in [0.05, 0.95]: Voronoi regions of mixtures of Gaussian-bump spectra."""
    dev = g.device

    def uni(*shape, lo=0.0, hi=1.0):
        return lo + (hi - lo) * torch.rand(*shape, generator=g, device=dev)

    R = regions or max(4, min(32, N1 * N2 // 2048))
    x = (torch.arange(N3, device=dev) + 0.5) / N3
    centre, width, amp = uni(endmembers, 3, 1), uni(endmembers, 3, 1, lo=0.05, hi=0.25), uni(endmembers, 3, 1, lo=0.2)
    E = (amp * torch.exp(-0.5 * ((x - centre) / width) ** 2)).sum(1)
    lo, hi = E.amin(1, keepdim=True), E.amax(1, keepdim=True)
    E = 0.05 + 0.9 * (E - lo) / (hi - lo).clamp_min(1e-6)
    A = -torch.log(uni(R, endmembers).clamp_min(1e-6))  # Dirichlet(1) by normalised exponentials
    A = A / A.sum(1, keepdim=True)
    si, sj = uni(R) * N1, uni(R) * N2
    ii, jj = torch.arange(N1, device=dev) + 0.5, torch.arange(N2, device=dev) + 0.5
    label = ((ii[:, None, None] - si) ** 2 + (jj[None, :, None] - sj) ** 2).argmin(2)
    return (A @ E)[label].contiguous()


def _observe(clean, g, sigma, p_s, p_t):
    """Gaussian noise, constant offsets on a share of each band's columns, then salt-and-pepper."""
    N1, N2, N3 = clean.shape
    v = clean + sigma * torch.randn(clean.shape, generator=g, device=clean.device)
    hit = torch.rand(N2, N3, generator=g, device=clean.device) < p_t
    v = v + hit * (torch.rand(N2, N3, generator=g, device=clean.device) - 0.5)
    r = torch.rand(clean.shape, generator=g, device=clean.device)
    return torch.where(r < p_s, (r < p_s / 2).to(v.dtype), v).contiguous()


def _radii(n, sigma, p_s, p_t):
    """eq. (RadiusSet) with rho = 0.95, in plain Python: (eps, alpha, beta)."""
    rho = 0.95
    return (rho * math.sqrt(sigma * sigma * n * (1 - p_s)) if sigma > 0 else 0.01, rho * n * p_s / 2,
            rho * 0.5 * n * p_t * (1 - p_s) / 2)


def _noisy(case, seed):
    g = _generator(seed)
    clean = _scene(case["N1"], case["N2"], case["N3"], g)
    return _observe(clean, g, case["sigma"], 0.05, case["p_t"])


def _batch_problems(case, seed):
    """The uneven cubes: shapes and noise levels from case["shapes"], contents from the seed."""
    sg = torch.Generator()
    sg.manual_seed(case["shapes"])

    def pick(*options):
        return options[int(torch.randint(len(options), (1,), generator=sg))]

    out = []
    for i in range(case["count"]):
        N1, N2 = (int(x) for x in torch.randint(case["lo"], case["hi"] + 1, (2,), generator=sg))
        N3, sigma, p_t, k = pick(31, 64, 128, 191), pick(0.05, 0.1), pick(0.0, 0.05, 0.1), pick(3, 5)
        v = _noisy({"N1": N1, "N2": N2, "N3": N3, "sigma": sigma, "p_t": p_t}, 1000 * seed + i)
        eps, alpha, beta = _radii(v.numel(), sigma, 0.05, p_t)
        out.append({"v": v, "eps": eps, "alpha": alpha, "beta": beta, "k": k})
    return out


def _net_params(seed):
    """He-normal weights, zero biases, a small head: the layout of the library's flat parameter vector."""
    g = _generator(seed + 77)
    parts = []
    for ci, co in NET_LAYERS:
        parts.append(torch.randn(co * 27 * ci, generator=g, device="cuda") * math.sqrt(2.0 / (27 * ci)))
        parts.append(torch.zeros(co, device="cuda"))
    parts.append(torch.randn(96, generator=g, device="cuda") * (0.1 / math.sqrt(32)))
    parts.append(torch.zeros(3, device="cuda"))
    return torch.cat(parts).contiguous()


def _crops(case, seed):
    """A batch of training crops: the observation and the targets (restored cube, sparse part, stripes)."""
    vs, us, ss, ts = [], [], [], []
    for i in range(case["batch"]):
        g = _generator(1000 * seed + i)
        clean = _scene(case["N1"], case["N2"], case["N3"], g)
        v = _observe(clean, g, 0.1, 0.05, 0.05)
        stripes = (v - clean).median(0, keepdim=True).values.expand_as(v)
        sparse = torch.where((v - clean - stripes).abs() > 0.3, v - clean - stripes, torch.zeros_like(v))
        for xs, x in zip((vs, us, ss, ts), (v, clean, sparse, stripes)):
            xs.append(x)
    return [torch.stack(xs).contiguous() for xs in (vs, us, ss, ts)]


# ---------------------------------------------------------------- the calls
def prepare(case, seed):
    kind = case["kind"]
    if kind == "quality":
        g = _generator(seed)
        ref = _scene(case["N1"], case["N2"], case["N3"], g)
        u = (ref + 0.02 * torch.randn(ref.shape, generator=g, device="cuda")).clamp_(0.0, 1.0)
        return {"kind": kind, "solver": P.Solver(), "u": u, "ref": ref}
    if kind in ("net", "train"):
        net = P.WarmStartNet()
        net.set_params(_net_params(seed))
        if kind == "net":
            return {"kind": kind, "net": net, "v": _noisy({**case, "sigma": 0.1, "p_t": 0.05}, seed)}
        return {"kind": kind, "net": net, "crops": _crops(case, seed),
                "grad": torch.empty(net.param_count, device="cuda")}
    solver = P.Solver()
    if kind == "batch":
        solver.set_option(B.OPT_STEP_POLICY, B.STEP_PC_EXACT)
        return {"kind": kind, "solver": solver, "problems": _batch_problems(case, seed), "passes": case["passes"]}
    v = _noisy(case, seed)
    eps, alpha, beta = _radii(v.numel(), case["sigma"], 0.05, case["p_t"])
    state = {"kind": kind, "solver": solver, "v": v, "passes": case["passes"], "k": case["k"],
             "radii": (eps, alpha, beta)}
    if kind == "resume":
        solver.set_option(B.OPT_STEP_POLICY, B.STEP_PC_EXACT)
        solver.setup(v, eps, alpha, beta, case["k"])
        return state
    if case["exact_steps"]:
        solver.set_option(B.OPT_STEP_POLICY, B.STEP_PC_EXACT)
    if case["stacked"]:
        solver.set_option(B.OPT_LAYOUT, B.LAYOUT_STACKED)
        solver.set_option(B.OPT_SPECTRAL_BOUNDARY, B.SPECTRAL_OPEN)
    solver.set_option(B.OPT_REGULARIZER, REGS[case["reg"]])
    return state


def run(state):
    kind = state["kind"]
    if kind == "solve":
        u, s, t, info = state["solver"].solve(state["v"], *state["radii"], state["k"], max_iter=state["passes"],
                                              tol=0.0)
        return {"u": u, "s": s, "t": t, "iters": info["iters"]}
    if kind == "resume":
        solver = state["solver"]
        info = solver.iterate(state["passes"])
        return {**{name: solver.get_state(name, like=state["v"]) for name in B.STATE}, "iters": info["iters"]}
    if kind == "batch":
        out = state["solver"].solve_batched(state["problems"], max_iter=state["passes"], tol=0.0)
        return [{"u": u, "s": s, "t": t, "iters": info["iters"]} for u, s, t, info in out]
    if kind == "net":
        return dict(zip(("u", "s", "t"), state["net"].forward(state["v"])))
    if kind == "train":
        loss, grad = state["net"].gradient(*state["crops"], grad=state["grad"])
        return {"loss": loss, "grad": grad}
    return state["solver"].quality(state["u"], state["ref"], sam_map=True)


# ---------------------------------------------------------------- what a pass cannot do without
def _solve_work(N1, N2, N3, k, passes, stacked=False, reg="s3ttv"):
    V = N1 * N2 * N3
    # u, s, t, y2, y3 read and written and v read; the two (block) dual parts read and written
    dual = 2 if reg == "sstv" else 2 * k * k
    n, w = (2 * k * k, N3) if stacked else (k * k, 2 * N3)
    flops = 60 * V if reg == "sstv" else 60 * V + N1 * N2 * (4 * n * n * w + 9 * n ** 3)
    return passes * (11 + 2 * dual) * 4 * V, passes * flops


def work(case):
    kind = case["kind"]
    if kind == "batch":
        sg = torch.Generator()
        sg.manual_seed(case["shapes"])
        by = fl = 0
        for _ in range(case["count"]):
            N1, N2 = (int(x) for x in torch.randint(case["lo"], case["hi"] + 1, (2,), generator=sg))
            picks = [int(torch.randint(n, (1,), generator=sg)) for n in (4, 2, 3, 2)]
            b, f = _solve_work(N1, N2, (31, 64, 128, 191)[picks[0]], (3, 5)[picks[3]], case["passes"])
            by, fl = by + b, fl + f
        return {"bytes": by, "flops": fl}
    V = case["N1"] * case["N2"] * case["N3"] * case.get("batch", 1)
    if kind == "quality":  # both cubes read once; the 11 x 11 window is separable: 5 moments of 22 taps
        return {"bytes": 8 * V + 4 * case["N1"] * case["N2"], "flops": (2 * 5 * 22 + 40) * V}
    if kind in ("net", "train"):
        mults = sum(27 * ci * co / 8 ** lvl for (ci, co), lvl in zip(NET_LAYERS, NET_LEVEL)) + 96
        if kind == "net":
            return {"bytes": 16 * V + 2 * 1411651, "flops": 2 * mults * V}
        return {"bytes": 16 * V + 6 * 1411651, "flops": 6 * mults * V}
    b, f = _solve_work(case["N1"], case["N2"], case["N3"], case["k"], case["passes"], case.get("stacked", False),
                       case.get("reg", "s3ttv"))
    if kind == "resume":  # the state read back
        b += (5 + 2 * case["k"] ** 2) * 8 * V
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------- the same in 64 bits
def _dif(x, axis):
    return torch.roll(x, -1, axis) - x


def _dif_t(x, axis):
    return torch.roll(x, 1, axis) - x


def _l1_ball(x, radius):
    a = x.abs().flatten()
    if float(a.sum()) <= radius:
        return x
    if radius <= 0:
        return torch.zeros_like(x)
    top = a.sort(descending=True).values
    over = (top.cumsum(0) - radius) / torch.arange(1, top.numel() + 1, device=x.device, dtype=x.dtype)
    tau = over[int((top > over).nonzero().max())]
    return x.sign() * (x.abs() - tau).clamp_min(0.0)


def _clip_blocks(Y):
    """Singular values of every Y[l] (n x w) clipped at 1."""
    out = torch.empty_like(Y)
    step = max(1, 200_000_000 // (Y.shape[1] * Y.shape[2]))
    for l in range(0, Y.shape[0], step):
        y = Y[l:l + step]
        lam, V = torch.linalg.eigh(y @ y.transpose(1, 2))
        f = torch.where(lam > 1, lam.clamp_min(1.0).rsqrt(), torch.ones_like(lam))
        out[l:l + step] = ((V * f[:, None, :]) @ V.transpose(1, 2)) @ y
    return out


def _ppds(v, radii, k, passes, exact_steps, stacked=False, reg="s3ttv"):
    """Alg. 1 from its usual start, in the precision of v; the state after `passes` passes."""
    eps, alpha, beta = radii
    N1, N2, N3 = v.shape
    gu = 1.0 / 9.0 if reg == "sstv" else 1.0 / (8.0 * k * k + 1) if exact_steps else 1.0 / (8.0 * N1 * N2 + 1)
    gs, gt, gY, g2, g3 = 1.0, 1.0 / 3.0, 0.25, 0.5, 1.0 / 3.0
    zero = torch.zeros_like
    u, s, t, y2, y3, Zv, Zh = v.clone(), zero(v), zero(v), zero(v), zero(v), zero(v), zero(v)
    n = k * k
    Y = torch.zeros((2, N1, N2, N3) if reg == "sstv" else (N1, N2, n, 2, N3), dtype=v.dtype, device=v.device)
    for _ in range(passes):
        x = u - gu * (_dif_t(_dif_t(Zv, 0) + _dif_t(Zh, 1), 2) + y3)
        un = x.clamp(0.0, 1.0)
        sn = _l1_ball(s - gs * y3, alpha)
        tn = _l1_ball(t - gt * (_dif_t(y2, 0) + y3), beta)
        ub, sb, tb = 2 * un - u, 2 * sn - s, 2 * tn - t
        u, s, t = un, sn, tn
        ds = _dif(ub, 2)
        if stacked:
            ds[:, :, -1] = 0.0
        fv, fh = _dif(ds, 0), _dif(ds, 1)
        if reg == "sstv":
            Y = (Y + gY * torch.stack((fv, fh))).clamp(-1.0, 1.0)
            Zv, Zh = Y[0], Y[1]
        else:
            for r in range(n):
                sh = (-(r // k), -(r % k))
                Y[:, :, r, 0] += gY * torch.roll(fv, sh, (0, 1))
                Y[:, :, r, 1] += gY * torch.roll(fh, sh, (0, 1))
            shape = (N1 * N2, 2 * n, N3) if stacked else (N1 * N2, n, 2 * N3)
            Y = _clip_blocks(Y.reshape(shape)).reshape(N1, N2, n, 2, N3)
            Zv, Zh = zero(v), zero(v)
            for r in range(n):
                sh = (r // k, r % k)
                Zv += torch.roll(Y[:, :, r, 0], sh, (0, 1))
                Zh += torch.roll(Y[:, :, r, 1], sh, (0, 1))
        y2 = y2 + g2 * _dif(tb, 0)
        y3p = y3 + g3 * (ub + sb + tb)
        d = y3p / g3 - v
        nd = float(d.norm())
        y3 = g3 * d * (1.0 - eps / nd) if nd > eps else zero(v)
    return {"u": u, "s": s, "t": t, "y2": y2, "y3": y3, "Y": Y}


def _net64(theta, v):
    """The network on a batch (B, D, H, W) in the precision of theta: (u, s, t)."""
    at = 0

    def take(*shape):
        nonlocal at
        at += math.prod(shape)
        return theta[at - math.prod(shape):at].reshape(shape)

    def conv(x):
        nonlocal layer
        ci, co = NET_LAYERS[layer]
        layer += 1
        w = take(co, 3, 3, 3, ci).permute(0, 4, 1, 2, 3)
        b = take(co)
        xp = F.pad(x, (1, 1, 1, 1, 1, 1))
        D, H, W = x.shape[2:]
        y = b.reshape(1, -1, 1, 1, 1).expand(x.shape[0], co, D, H, W)
        for tap in range(27):
            dz, dy, dx = tap // 9, tap // 3 % 3, tap % 3
            y = y + torch.einsum("oc,bczyx->bozyx", w[:, :, dz, dy, dx],
                                 xp[:, :, dz:dz + D, dy:dy + H, dx:dx + W])
        return F.relu(y)

    def up(x):
        return x.repeat_interleave(2, 2).repeat_interleave(2, 3).repeat_interleave(2, 4)

    layer = 0
    x = v[:, None]
    e1 = conv(conv(x))
    e2 = conv(conv(F.avg_pool3d(e1, 2)))
    b = conv(conv(F.avg_pool3d(e2, 2)))
    d2 = conv(conv(torch.cat((up(b), e2), 1)))
    d1 = conv(conv(torch.cat((up(d2), e1), 1)))
    w, bias = take(3, 32), take(3)
    h = torch.einsum("jc,bczyx->jbzyx", w, d1) + bias.reshape(3, 1, 1, 1, 1)
    return v + h[0], h[1], h[2]


def _quality64(u, ref, trim=3):
    N1, N2, N3 = u.shape
    b = slice(trim, N3 - trim) if N3 > 2 * trim else slice(0, N3)
    mse = ((u - ref) ** 2).mean((0, 1))[b]
    out = {"mpsnr": float((-10.0 * mse.log10()).mean())}
    a = torch.arange(-5, 6, device=u.device, dtype=u.dtype)
    w1 = torch.exp(-a * a / (2 * 1.5 * 1.5))
    w1 = w1 / w1.sum()

    def mean(x):  # the 11 x 11 Gaussian window over the pixels that hold it whole
        x = sum(w1[i] * x[i:N1 - 10 + i] for i in range(11))
        return sum(w1[i] * x[:, i:N2 - 10 + i] for i in range(11))

    x, y = ref[:, :, b], u[:, :, b]
    mx, my = mean(x), mean(y)
    sx, sy, sxy = mean(x * x) - mx * mx, mean(y * y) - my * my, mean(x * y) - mx * my
    ssim = (2 * mx * my + 1e-4) * (2 * sxy + 9e-4) / ((mx * mx + my * my + 1e-4) * (sx + sy + 9e-4))
    out["mssim"] = float(ssim.mean())
    c = (u * ref).sum(2) / (u.norm(dim=2) * ref.norm(dim=2))
    out["sam_map"] = c.clamp(-1.0, 1.0).acos()
    out["sam"] = float(out["sam_map"].mean())
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "quality":
        s = prepare(case, seed)
        return _quality64(s["u"].double(), s["ref"].double())
    V = case["N1"] * case["N2"] * case["N3"] * case.get("batch", 1) if kind != "batch" else 0
    if kind == "net":
        if V > 1 << 20:
            return None  # minutes in 64 bits
        v = _noisy({**case, "sigma": 0.1, "p_t": 0.05}, seed).double()
        with torch.no_grad():
            u, s, t = _net64(_net_params(seed).double(), v[None])
        return {"u": u[0], "s": s[0], "t": t[0]}
    if kind == "train":
        if V > 1 << 18:
            return None
        v, tu, ts, tt = (x.double() for x in _crops(case, seed))
        theta = _net_params(seed).double().requires_grad_()
        loss = sum(((a - b) ** 2).sum() for a, b in zip(_net64(theta, v), (tu, ts, tt))) / (3 * v.numel())
        (grad,) = torch.autograd.grad(loss, theta)
        return {"loss": float(loss.detach()), "grad": grad}
    if kind == "batch":
        return None  # each member is what solve gives alone
    k, sstv = case["k"], case.get("reg", "s3ttv") == "sstv"
    n = 2 * k * k if case.get("stacked") else k * k
    # the eigen-solves in 64 bits: batched on the GPU up to 32 rows (13 s at 4.1e10), one by one above (minutes)
    if not sstv and case["N1"] * case["N2"] * case["passes"] * n ** 3 > (4.5e10 if n <= 32 else 1e8):
        return None
    v = _noisy(case, seed).double()
    st = _ppds(v, _radii(v.numel(), case["sigma"], 0.05, case["p_t"]), k, case["passes"],
               kind == "resume" or case["exact_steps"], case.get("stacked", False), case.get("reg", "s3ttv"))
    if kind == "solve":
        return {"u": st["u"], "s": st["s"], "t": st["t"], "iters": None}
    # the external order of the block duals: column 2b + o
    Y = st["Y"].transpose(3, 4).reshape(case["N1"] * case["N2"], k * k, 2 * case["N3"])
    return {**{name: st[name] for name in ("u", "s", "t", "y2", "y3")}, "Y": Y, "iters": None}
