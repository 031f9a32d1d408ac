"""The workloads whose speed is watched, as a user's program runs them.

Every case is one restoration (or one layer of the warm-start network, trained)
through the package's public entry points, from a cold or warm start to the
posterior mean and marginal variance.  A program that restores images keeps one
context per problem size and operator (``EPTV``, ``Batch``, ``WarmStartNet``), so
the context is prepared and a pass re-initialises its sites, sweeps, and reads
the posterior; ``solve`` cases make the whole call from host memory, context
included.

Sizes and parameters are those of the package's configurations and tests
(``bench.py``, ``synthetic.py``, ``tests/``): denoising from 64^2 to 4096^2 with
odd and free-boundary sizes and the mixture prior, deconvolution of 9x9 uniform
and 15x15 Gaussian blurs on power-of-two and ragged sizes, an uneven batch,
compressive sensing with dense and Hadamard rows, and the network.

``exact`` computes the same results with torch in 64 bits, from the formulas of
Yao, McLaughlin and Altmann (arXiv:2110.01585), without the library.
"""
import ctypes
import math
import os

import numpy as np
import torch

import paper_2110_01585_gb300 as eptv
from paper_2110_01585_gb300 import _lib
from paper_2110_01585_gb300 import synthetic as syn
from paper_2110_01585_gb300.warmstart import WarmStartNet

DAMPING = 0.5
VAR_CAP = 1e8
PROBE_SEED = 1234
MOG2 = (0.3, 0.1, 1e-4)  # omega, s1^2, s2^2
NET_FILE = os.path.join(os.path.dirname(eptv.__file__), "data", "warmstart_gauss15_128.npz")
NET_BLUR_STD = 2.0


def listed():
    return [
        # the smallest restoration: 64^2, sigma 0.1, 50 sweeps; one short launch after another
        dict(name="denoise_64", kind="denoise", h=64, w=64, sigma=0.1, beta=20.0, sweeps=50, em=0,
             periodic=True, prior="l1", noise="iid"),
        # an ordinary image whose TV parameter is estimated along the way
        dict(name="denoise_512_em", kind="denoise", h=512, w=512, sigma=0.1, beta=1.0, sweeps=20, em=5,
             periodic=True, prior="l1", noise="iid"),
        # the largest image: the prior pass streams 16.8 M pixels per sweep
        dict(name="denoise_4096", kind="denoise", h=4096, w=4096, sigma=0.1, beta=20.0, sweeps=5, em=0,
             periodic=True, prior="l1", noise="iid"),
        # odd sides, free boundary, the Gaussian-mixture prior
        dict(name="denoise_mog2_611x777", kind="denoise", h=611, w=777, sigma=0.1, beta=0.0, sweeps=20,
             em=0, periodic=False, prior="mog2", noise="iid"),
        # deconvolution as the package is benched: 9x9 blur, BSNR 40 dB, EM every 5 sweeps
        dict(name="deconv_512", kind="deconv", h=512, w=512, blur="uniform", width=9, bsnr=40.0,
             probes=32, sweeps=10, em=5),
        # an image whose sides are not powers of two
        dict(name="deconv_300x420", kind="deconv", h=300, w=420, blur="uniform", width=9, bsnr=30.0,
             probes=32, sweeps=5, em=5),
        # network prediction, warm start and EP sweeps: 15x15 Gaussian blur, BSNR 30 dB
        dict(name="warm_256", kind="warm", h=256, w=256, probes=32, sweeps=10),
        # many uneven problems advanced together
        dict(name="batch_32", kind="batch", n=32, min_side=64, max_side=512, sweeps=3, em=0),
        # compressive sensing, dense Gaussian rows (M = 0.3 N)
        dict(name="cs_dense_64", kind="cs", op="dense", side=64, m=1228, sigma=0.01, sweeps=5, em=5),
        # single-pixel imaging: M = 0.3 N Hadamard patterns
        dict(name="cs_hadamard_128", kind="cs", op="hadamard", side=128, m=4915, sigma=0.01, sweeps=2,
             em=0),
        # a hidden layer of the network in a training step: its forward pass, and the
        # gradients of its input, weights and bias, on a minibatch
        dict(name="net_layer_8x128", kind="layer", n=8, cin=32, cout=32, h=128, w=128, relu=True),
        # one restoration from host memory to host memory, context created and freed
        dict(name="solve_host_256", kind="solve", h=256, w=256, blur="uniform", width=9, bsnr=40.0,
             probes=32, sweeps=5, em=5),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["denoise", "denoise", "deconv", "deconv", "warm", "batch", "cs", "layer", "solve"])
    if kind == "denoise":
        h, w = _log_int(rng, 48, 4096), _log_int(rng, 48, 4096)
        prior = rng.choice(["l1", "l1", "mog2"])
        periodic = rng.random() < 0.6
        if periodic:
            h, w = h + h % 2, w + w % 2
        return dict(kind=kind, h=min(h, 4096), w=min(w, 4096), sigma=round(rng.uniform(0.05, 0.2), 3),
                    beta=round(rng.uniform(5.0, 25.0), 2) if prior == "l1" else 0.0,
                    sweeps=rng.randint(3, 5) if h * w > 1 << 21 else rng.randint(5, 40),
                    em=rng.choice([0, 5]) if prior == "l1" else 0, periodic=periodic, prior=prior,
                    noise=rng.choice(["iid", "iid", "plane"]))
    if kind in ("deconv", "solve"):
        if rng.random() < 0.4:
            h = w = rng.choice([64, 128, 256, 512])
        else:
            h, w = 2 * _log_int(rng, 24, 240), 2 * _log_int(rng, 24, 240)
        blur = rng.choice(["uniform", "uniform", "random"])
        return dict(kind=kind, h=h, w=w, blur=blur, width=rng.choice([5, 9]) if blur == "uniform" else 5,
                    bsnr=rng.choice([30.0, 40.0]), probes=rng.choice([16, 32]), sweeps=rng.randint(3, 8),
                    em=rng.choice([0, 5]))
    if kind == "warm":
        return dict(kind=kind, h=rng.choice([64, 128, 192, 256, 300, 384]),
                    w=rng.choice([64, 128, 200, 256, 320, 512]), probes=32, sweeps=rng.randint(4, 12))
    if kind == "batch":
        return dict(kind=kind, n=rng.randint(4, 32), min_side=64, max_side=rng.choice([128, 256, 512]),
                    sweeps=rng.randint(2, 3), em=rng.choice([0, 2]))
    if kind == "cs":
        op = rng.choice(["dense", "hadamard"])
        side = rng.choice([16, 32, 64]) if op == "hadamard" else rng.randint(16, 80)
        return dict(kind=kind, op=op, side=side, m=int(rng.uniform(0.2, 0.5) * side * side), sigma=0.01,
                    sweeps=rng.randint(2, 5), em=rng.choice([0, 2]))
    return dict(kind=kind, n=rng.randint(1, 16), cin=rng.choice([3, 32, 32]), cout=rng.choice([6, 32, 32]),
                h=rng.choice([64, 100, 128, 150]), w=rng.choice([64, 97, 128, 200]), relu=rng.random() < 0.8)


# ------------------------------------------------------------------- inputs

_STREAM = None


def _stream():
    """The one stream that the program works on."""
    global _STREAM
    if _STREAM is None:
        _STREAM = torch.cuda.Stream()
    return _STREAM


def _cuda(a):
    return torch.as_tensor(np.asarray(a, np.float32), device="cuda")


def _denoise_inputs(case, seed):
    p = syn.denoise_problem(case["h"], case["w"], sigma=case["sigma"], beta=case["beta"], seed=seed,
                            n_rect=8 if case["h"] * case["w"] < 1 << 20 else 40)
    y, xi = p.y.astype(np.float32), p.xi
    plane = None
    if case["noise"] == "plane":
        # per-pixel variances xi exp(U[0, 3]), the noise drawn accordingly
        rng = np.random.default_rng(seed + 77)
        plane = (0.4 * xi * np.exp(rng.uniform(0.0, 3.0, size=p.shape))).astype(np.float32)
        y = (p.x + np.sqrt(plane) * rng.standard_normal(p.shape)).astype(np.float32)
    return y, xi, plane


def _kernel(case, seed):
    if case["blur"] == "uniform":
        return syn.uniform_kernel(case["width"])
    # a full-rank (non-separable) kernel with more rows than columns
    rng = np.random.default_rng(seed + 5)
    k = rng.uniform(0.1, 1.0, size=(case["width"], case["width"] - 2))
    return k / k.sum()


def _deconv_inputs(case, seed):
    return syn.deconv_problem(case["h"], case["w"], kernel=_kernel(case, seed), bsnr_db=case["bsnr"], beta0=1.0,
                              seed=seed, grf_length=min(case["h"], case["w"]) / 16.0)


def _net_meta():
    meta = np.load(NET_FILE)
    return float(meta["beta"])


def _warm_inputs(case, seed):
    return syn.warmstart_problem(case["h"], case["w"], seed=seed, beta=_net_meta())


def _cs_inputs(case, seed):
    """(y, A or None, patterns or None): A on the GPU in FP32."""
    side, m, n = case["side"], case["m"], case["side"] ** 2
    rng = np.random.default_rng(seed)
    x = syn.piecewise_image(side, side, rng, n_rect=8, n_disc=4, grf_length=max(1.0, side / 16.0))
    noise = case["sigma"] * rng.standard_normal(m)
    if case["op"] == "dense":
        g = torch.Generator(device="cuda")
        g.manual_seed(seed)
        A = torch.randn((m, n), generator=g, device="cuda", dtype=torch.float32) / math.sqrt(m)
        y = (A.double() @ torch.as_tensor(x.reshape(-1), device="cuda")).cpu().numpy() + noise
        return y.astype(np.float32), A, None
    patterns = np.sort(rng.choice(n, size=m, replace=False)).astype(np.int32)
    A = _hadamard_rows(patterns, side)
    y = (A @ torch.as_tensor(x.reshape(-1), device="cuda")).cpu().numpy() + noise
    return y.astype(np.float32), None, patterns


def _hadamard_rows(patterns, side):
    """The M Paley-ordered patterns over sqrt(M), in 64 bits on the GPU."""
    bits = side.bit_length() - 1

    def walsh():
        """[k, r] = (-1)^popcount(r & rev(k)), rev reversing the index bits."""
        k = torch.arange(side, device="cuda")
        rev = torch.zeros_like(k)
        for b in range(bits):
            rev |= ((k >> b) & 1) << (bits - 1 - b)
        v = k[None, :] & rev[:, None]
        par = torch.zeros_like(v)
        for b in range(bits):
            par ^= (v >> b) & 1
        return (1 - 2 * par).double()

    wm = walsh()
    p = torch.as_tensor(patterns, device="cuda", dtype=torch.int64)
    rows = wm[p // side][:, :, None] * wm[p % side][:, None, :]
    return rows.reshape(len(patterns), side * side) / math.sqrt(len(patterns))


def _batch_inputs(case, seed):
    """Sides log-uniform and blur widths {1, 5, 9, 15} (1: denoising), the same for
    every seed; images and noise levels U[0.02, 0.2] by the seed."""
    plan, rng = np.random.default_rng([case["n"], case["max_side"]]), np.random.default_rng(seed)
    out = []
    for _ in range(case["n"]):
        side = int(round(math.exp(plan.uniform(math.log(case["min_side"]), math.log(case["max_side"])))))
        side += side % 2
        width = int(plan.choice([1, 5, 9, 15]))
        sigma, sub = float(rng.uniform(0.02, 0.2)), int(rng.integers(0, 2 ** 31))
        if width == 1:
            out.append(syn.denoise_problem(side, side, sigma=sigma, beta=1.0, seed=sub))
        else:
            out.append(syn.deconv_problem(side, side, kernel=syn.uniform_kernel(width), sigma=sigma, seed=sub,
                                          grf_length=side / 16.0))
    return out


def _layer_inputs(case, seed):
    """One layer as a training step meets it: activations x >= 0 of the layer before,
    He-scaled weights, the gradient dy of its output, and its output saved by the
    forward pass, which the backward pass reads for the ReLU's mask."""
    n, cin, cout, h, w = (case[k] for k in ("n", "cin", "cout", "h", "w"))
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)

    def normal(*shape):
        return torch.randn(shape, generator=g, device="cuda", dtype=torch.float32)

    x, wt = torch.relu(normal(n, cin, h, w)), normal(cout, cin, 3, 3) * math.sqrt(2.0 / (9 * cin))
    b, dy = 0.1 * normal(cout), normal(n, cout, h, w)
    saved = torch.relu(_conv64(x.double(), wt.double(), b.double())).float() if case["relu"] else None
    return x, wt, b, dy, saved


# ----------------------------------------------------------------- the passes

def _context(case, seed):
    kind, st = case["kind"], _stream()
    if kind == "denoise":
        y, xi, plane = _denoise_inputs(case, seed)
        kw = {}
        if case["prior"] == "mog2":
            kw = dict(prior=eptv.PRIOR_MOG2, omega=MOG2[0], s1_sq=MOG2[1], s2_sq=MOG2[2])
        return eptv.EPTV(_cuda(y), xi, case["beta"], stream=st, periodic=int(case["periodic"]),
                         xi_plane=None if plane is None else _cuda(plane), **kw)
    if kind in ("deconv", "warm"):
        p = _deconv_inputs(case, seed) if kind == "deconv" else _warm_inputs(case, seed)
        return eptv.EPTV(_cuda(p.y), p.xi, p.beta, op=eptv.OP_CONV_PERIODIC, kernel=p.kernel,
                         rbmc_samples=case["probes"], cg_max_iter=100000, stream=st)
    y, A, patterns = _cs_inputs(case, seed)
    kw = dict(op=eptv.OP_DENSE, dense=A) if A is not None else dict(op=eptv.OP_HADAMARD, patterns=patterns)
    return eptv.EPTV(_cuda(y), case["sigma"] ** 2, 1.0, height=case["side"], width=case["side"], stream=st, **kw)


def prepare(case, seed):
    kind, st = case["kind"], _stream()
    state = dict(case=dict(case))
    with torch.cuda.stream(st):
        if kind == "batch":
            state["eps"] = []
            for p in _batch_inputs(case, seed):
                kw = {} if p.kind == "denoise" else dict(op=eptv.OP_CONV_PERIODIC, kernel=p.kernel, rbmc_samples=32,
                                                         cg_max_iter=100000)
                state["eps"].append(eptv.EPTV(_cuda(p.y), p.xi, p.beta, stream=st, **kw))
            state["batch"] = eptv.Batch(state["eps"])
        elif kind == "layer":
            state["io"] = _layer_inputs(case, seed)
            state["lib"] = _lib.load()
        elif kind == "solve":
            p = _deconv_inputs(case, seed)
            state.update(y=p.y.astype(np.float32), xi=p.xi, kernel=p.kernel)
        else:
            state["ep"] = _context(case, seed)
            if kind == "warm":
                p = _warm_inputs(case, seed)
                net, _ = WarmStartNet.load(NET_FILE)
                net.stream = st
                state.update(net=net, y=_cuda(p.y), xi=p.xi)
    return state


def _layer(state):
    """Forward and backward of one 3x3 convolution through the C interface."""
    lib, (x, wt, b, dy, saved) = state["lib"], state["io"]
    n, cin, cout, h, w = (state["case"][k] for k in ("n", "cin", "cout", "h", "w"))
    ptr = lambda t: ctypes.c_void_p(None if t is None else t.data_ptr())  # noqa: E731
    stream = ctypes.c_void_p(_stream().cuda_stream)
    y, dx, dw, db = torch.empty_like(dy), torch.empty_like(x), torch.empty_like(wt), torch.empty_like(b)
    work_bytes = lib.ep_tv_conv3x3_backward_work(n, cin, cout, h, w)
    scratch = torch.empty(work_bytes, dtype=torch.uint8, device="cuda")
    _lib.check(lib.ep_tv_conv3x3_forward(n, cin, cout, h, w, ptr(x), ptr(wt), ptr(b), int(state["case"]["relu"]),
                                         ptr(y), stream), "ep_tv_conv3x3_forward")
    _lib.check(lib.ep_tv_conv3x3_backward(n, cin, cout, h, w, ptr(x), ptr(wt), ptr(saved), ptr(dy), ptr(dx),
                                          ptr(dw), ptr(db), ptr(scratch), ctypes.c_size_t(work_bytes), stream),
               "ep_tv_conv3x3_backward")
    return dict(y=y, dx=dx, dw=dw, db=db)


def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind == "solve":
        mean, var, beta = eptv.solve_host(state["y"], state["xi"], 1.0, case["sweeps"], case["em"],
                                          op=eptv.OP_CONV_PERIODIC, kernel=state["kernel"],
                                          rbmc_samples=case["probes"], cg_max_iter=100000)
        return dict(mean=mean, var=var, beta=beta)
    with torch.cuda.stream(_stream()):
        if kind == "batch":
            for ep in state["eps"]:
                ep.reset()
            state["batch"].sweep(case["sweeps"], em_every=case["em"])
            # one tensor of all images, each flattened
            post = [ep.posterior() for ep in state["eps"]]
            return dict(mean=torch.cat([m.reshape(-1) for m, _ in post]),
                        var=torch.cat([v.reshape(-1) for _, v in post]))
        if kind == "layer":
            return _layer(state)
        ep = state["ep"]
        ep.reset()
        if kind == "warm":
            eptv.warm_start(ep, state["net"].predict(state["y"], state["xi"], NET_BLUR_STD))
            ep.sweep(case["sweeps"])
        else:
            ep.sweep(case["sweeps"], em_every=case["em"])
        mean, var = ep.posterior()
        res = dict(mean=mean, var=var)
        if case.get("em") and case["sweeps"] % case["em"] == 0:
            res["beta"] = ep.em_beta()[0]  # the statistic of the last sweep, whose EM step set beta
        return res


# ------------------------------------------------------------- minimal work

def work(case):
    """Bytes: y in, mean and variance out, and per sweep the five sites (the prior
    ones read and written, the likelihood site read, for deconvolution also
    written) and the solver's FP64 solutions (read and written), or A for dense
    sensing.  Flops: 150 per edge update (four per two pixels); deconvolution 20
    conjugate-gradient iterations per sweep and system, each two real 2-D
    transforms (2.5 N log2 N each) and 20 N; sensing K = A C A^T, its Cholesky
    factor and inverse, and W = L^-1 A; the network 18 cin cout per pixel
    and layer, three times that with the gradients."""
    def image(n, sweeps, conv, probes):
        b = 12.0 * n + sweeps * n * (72.0 if conv else 68.0)
        f = sweeps * 300.0 * n
        if conv:
            r = 1 + probes
            b += sweeps * n * (16.0 * r + 8.0)
            f += sweeps * 20.0 * r * n * (5.0 * math.log2(n) + 20.0)
        return b, f

    net = 18.0 * (3 * 32 + 4 * 32 * 32 + 32 * 6)
    kind = case["kind"]
    if kind == "denoise":
        b, f = image(case["h"] * case["w"], case["sweeps"], False, 0)
    elif kind in ("deconv", "solve", "warm"):
        n = case["h"] * case["w"]
        b, f = image(n, case["sweeps"], True, case["probes"])
        if kind == "warm":
            b, f = b + 4.0 * n * 7, f + net * n
    elif kind == "batch":
        # sides log-uniform: E[side^2]; three problems in four are blurred
        lo, hi = case["min_side"], case["max_side"]
        n = (hi * hi - lo * lo) / (2.0 * math.log(hi / lo))
        b1, f1 = image(n, case["sweeps"], True, 32)
        b0, f0 = image(n, case["sweeps"], False, 0)
        b, f = case["n"] * (0.75 * b1 + 0.25 * b0), case["n"] * (0.75 * f1 + 0.25 * f0)
    elif kind == "cs":
        n, m = float(case["side"] ** 2), float(case["m"])
        b, f = image(n, case["sweeps"], False, 0)
        dense = case["op"] == "dense"
        b += case["sweeps"] * 4.0 * m * (n if dense else 1.0)
        # symmetric K and triangular L^-1 halve the dense products; transforms otherwise
        f += case["sweeps"] * (2.0 / 3.0 * m ** 3 + (2.0 * m * m * n if dense else 2.0 * m * n * math.log2(n)))
    else:
        n, cin, cout = float(case["n"] * case["h"] * case["w"]), case["cin"], case["cout"]
        b = 4.0 * n * (2 * cin + 3 * cout) + 4.0 * (2 * 9 * cin * cout + 2 * cout)
        f = 3.0 * 18.0 * cin * cout * n
    return dict(bytes=b, flops=f)


# --------------------------------------------- the same in 64 bits (plain torch)

def _mills(a):
    """g = h - a and v = 1 - h g of a standard normal truncated to [a, inf): the
    closed form with erfcx, and for a > 5 Laplace's continued fraction."""
    lo = torch.clamp(a, max=5.0)
    h = math.sqrt(2.0 / math.pi) / torch.special.erfcx(lo / math.sqrt(2.0))
    g, v = h - lo, 1.0 - h * (h - lo)
    big = a > 5.0
    if bool(big.any()):
        ab = torch.clamp(a, min=5.0)
        t = torch.zeros_like(ab)
        t2 = t
        for k in range(64, 0, -1):
            t = k / (ab + t)
            if k == 2:
                t2 = t
        g = torch.where(big, t, g)
        v = torch.where(big, t * (t2 - t), v)
    return g, v


def _log_erfcx(x):
    """log erfcx, also where erfcx overflows (erfcx(x) = exp(x^2) erfc(x))."""
    far = x < -20.0
    return torch.where(far, x * x + torch.log(torch.special.erfc(torch.clamp(x, max=0.0))),
                       torch.log(torch.special.erfcx(torch.clamp(x, min=-20.0))))


def _tilted_l1(mu, s2, lam):
    s = torch.sqrt(s2)
    ap, am = lam * s - mu / s, lam * s + mu / s
    d = _log_erfcx(am / math.sqrt(2.0)) - _log_erfcx(ap / math.sqrt(2.0))
    wp, wm = torch.sigmoid(-d), torch.sigmoid(d)
    gp, vp = _mills(ap)
    gm, vm = _mills(am)
    ep, em = s * gp, -s * gm
    return wp * ep + wm * em, wp * s2 * vp + wm * s2 * vm + wp * wm * (ep - em) ** 2, wp * ep - wm * em


def _tilted_mog2(mu, s2):
    om, v1, v2 = MOG2
    e1, e2 = v1 + s2, v2 + s2
    l1 = math.log(om) - 0.5 * torch.log(e1) - mu ** 2 / (2 * e1)
    l2 = math.log(1 - om) - 0.5 * torch.log(e2) - mu ** 2 / (2 * e2)
    w1, w2 = torch.sigmoid(l1 - l2), torch.sigmoid(l2 - l1)
    m1, m2 = mu * v1 / e1, mu * v2 / e2
    var = w1 * v1 * s2 / e1 + w2 * v2 * s2 / e2 + w1 * w2 * (m1 - m2) ** 2
    return w1 * m1 + w2 * m2, var, torch.zeros_like(mu)


class _EP64:
    """The damped sweep of Algorithm 1 on an image, sites in natural parameters."""

    def __init__(self, h, w, tau0, nu0, beta, site0=None, periodic=True, prior="l1"):
        self.h, self.w, self.beta, self.site0, self.prior = h, w, beta, site0, prior
        self.tau = torch.full((5, h, w), 1.0 / VAR_CAP, dtype=torch.float64, device="cuda")
        self.nu = torch.zeros((5, h, w), dtype=torch.float64, device="cuda")
        self.tau[0], self.nu[0] = tau0, nu0

        def pairs(n, first):
            i = torch.arange(first, n, 2, device="cuda")
            return (i, (i + 1) % n) if periodic else (i[i + 1 < n], i[i + 1 < n] + 1)

        self.pairs = [(1, pairs(w, 0)), (1, pairs(w, 1)), (0, pairs(h, 0)), (0, pairs(h, 1))]

    def _prior_site(self, k):
        dim, (i, j) = self.pairs[k - 1]
        if not len(i):
            return 0.0
        tc = self.tau.sum(0) - self.tau[k]
        nc = self.nu.sum(0) - self.nu[k]
        ti, tj, ni, nj = (x.index_select(dim, y) for x, y in ((tc, i), (tc, j), (nc, i), (nc, j)))
        ci, cj = 1.0 / ti, 1.0 / tj
        mi, mj = ni * ci, nj * cj
        mu, s2 = mi - mj, ci + cj
        mb, sb, eab = _tilted_l1(mu, s2, self.beta) if self.prior == "l1" else _tilted_mog2(mu, s2)
        for idx, c, m, t, n, sg in ((i, ci, mi, ti, ni, 1.0), (j, cj, mj, tj, nj, -1.0)):
            e = m + sg * (mb - mu) / s2 * c
            var = c + (sb - s2) / s2 ** 2 * c ** 2
            tn = torch.clamp(1.0 / var - t, min=1.0 / VAR_CAP)
            nn = (tn + t) * e - n
            for site, new in ((self.tau[k], tn), (self.nu[k], nn)):
                old = site.index_select(dim, idx)
                site.index_copy_(dim, idx, DAMPING * new + (1.0 - DAMPING) * old)
        return float(eab.sum())

    def sweep(self, n, em=0):
        for t in range(n):
            a = sum(self._prior_site(k) for k in (1, 2, 3, 4))
            if self.site0 is not None:
                d, nc = self.tau[1:].sum(0), self.nu[1:].sum(0)
                e, var = self.site0(d, nc)
                tn = torch.clamp(1.0 / var - d, min=1.0 / VAR_CAP)
                nn = (tn + d) * e - nc
                self.tau[0] = DAMPING * tn + (1.0 - DAMPING) * self.tau[0]
                self.nu[0] = DAMPING * nn + (1.0 - DAMPING) * self.nu[0]
            if em and (t + 1) % em == 0:
                self.beta = self.h * self.w / a

    def posterior(self):
        t = self.tau.sum(0)
        return self.nu.sum(0) / t, 1.0 / t


def _f64(a):
    return torch.as_tensor(np.asarray(a, np.float32), device="cuda").double()


def _normals(count, base):
    """Draws base, base + 1, ... of the library's documented probe stream: SplitMix64
    as a counter-based generator, two 24-bit uniforms, Box-Muller; kept in FP32."""
    t = 2 * (base + np.arange(count, dtype=np.uint64))

    def mix(t):
        z = np.uint64(PROBE_SEED) + (t + np.uint64(1)) * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return ((z ^ (z >> np.uint64(31))) >> np.uint64(40)).astype(np.float64)

    with np.errstate(over="ignore"):
        u1 = (mix(t) + 0.5) / 16777216.0
        u2 = (mix(t + np.uint64(1)) + 0.5) / 16777216.0
    return (np.sqrt(-2.0 * np.log(u1)) * np.cos(6.283185307179586 * u2)).astype(np.float32)


class _Deconv64:
    """Likelihood site of a periodic blur: the mean and S probe systems of
    Q = H^T H / xi + diag(d) by circulant-preconditioned conjugate gradients."""

    def __init__(self, y, xi, kernel, probes):
        h, w = y.shape
        k = np.asarray(kernel, np.float32).astype(np.float64)
        pad = np.zeros((h, w))
        pad[:k.shape[0], :k.shape[1]] = k
        pad = np.roll(pad, (-(k.shape[0] // 2), -(k.shape[1] // 2)), axis=(0, 1))
        self.hf = torch.fft.rfft2(torch.as_tensor(pad, device="cuda"))
        self.hth = self.hf.abs() ** 2
        self.xi, self.g0 = xi, float((k * k).sum()) / xi
        n = h * w
        e1 = _f64(_normals(probes * n, 0)).reshape(probes, h, w)
        e2 = _f64(_normals(probes * n, probes * n)).reshape(probes, h, w)
        self.hw = (h, w)
        self.hty = self._ht(_f64(y)) / xi
        self.e1, self.e2 = self._ht(e1) / math.sqrt(xi), e2
        self.x = None

    def _ht(self, v):
        return torch.fft.irfft2(torch.fft.rfft2(v) * self.hf.conj(), s=self.hw)

    def _filter(self, v, f):
        return torch.fft.irfft2(torch.fft.rfft2(v) * f, s=self.hw)

    def __call__(self, d, nc):
        b = torch.cat([(self.hty + nc)[None], self.e1 + torch.sqrt(d) * self.e2])
        f = 1.0 / (self.hth / self.xi + d.mean())
        q = lambda v: self._filter(v, self.hth / self.xi) + d * v  # noqa: E731
        dot = lambda u, v: (u * v).sum((1, 2), keepdim=True)  # noqa: E731
        x = torch.zeros_like(b) if self.x is None else self.x
        r = b - q(x)
        stop = 1e-24 * dot(b, b)
        z = self._filter(r, f)
        p, rz = z, dot(r, z)
        for it in range(4000):
            if it % 10 == 0 and bool((dot(r, r) <= stop).all()):
                break
            ap = q(p)
            al = rz / torch.clamp(dot(p, ap), min=1e-300)
            x = x + al * p
            r = r - al * ap
            z = self._filter(r, f)
            rz2 = dot(r, z)
            p = z + rz2 / torch.clamp(rz, min=1e-300) * p
            rz = rz2
        self.x = x
        off = self._filter(x[1:], self.hth / self.xi) - self.g0 * x[1:]
        minv = 1.0 / (self.g0 + d)
        return x[0], minv + minv ** 2 * (off ** 2).mean(0)


def _cs64(A, y, xi):
    def site0(d, nc):
        shape = d.shape
        c, m = (1.0 / d).reshape(-1), (nc / d).reshape(-1)
        K = (A * c) @ A.T
        K.diagonal().add_(xi)
        L = torch.linalg.cholesky(K)
        wv = (torch.linalg.solve_triangular(L, A, upper=False) ** 2).sum(0)
        u = torch.cholesky_solve((y - A @ m)[:, None], L)[:, 0]
        return (m + c * (A.T @ u)).reshape(shape), (c - c * c * wv).reshape(shape)
    return site0


def _conv64(x, w, b):
    x = torch.nn.functional.pad(x, (1, 1, 1, 1), mode="circular")
    return torch.nn.functional.conv2d(x, w, b)


def _net64(x, params):
    for i, (w, b) in enumerate(params):
        x = _conv64(x, w, b)
        if i + 1 < len(params):
            x = torch.relu(x)
    return x


def _features64(y, xi):
    x = torch.empty((y.shape[0], 3) + tuple(y.shape[1:]), dtype=torch.float64, device="cuda")
    x[:, 0] = y
    x[:, 1] = _f64(np.log10(xi) / 4.0).view(-1, 1, 1)
    x[:, 2] = NET_BLUR_STD / 4.0
    return x


def exact(case, seed):
    kind = case["kind"]
    if kind == "layer":
        x, wt, b, dy, saved = _layer_inputs(case, seed)
        x, wt, b = (t.double().requires_grad_(True) for t in (x, wt, b))
        z = _conv64(x, wt, b)
        g = dy.double() if saved is None else torch.where(saved > 0, dy, torch.zeros_like(dy)).double()
        dx, dw, db = torch.autograd.grad(z, (x, wt, b), g)
        return dict(y=(torch.relu(z) if case["relu"] else z).detach(), dx=dx, dw=dw, db=db)
    if kind == "denoise":
        y, xi, plane = _denoise_inputs(case, seed)
        v = xi if plane is None else _f64(plane)
        ep = _EP64(case["h"], case["w"], 1.0 / v, _f64(y) / v, case["beta"], periodic=case["periodic"],
                   prior=case["prior"])
    elif kind == "batch":
        post = []
        for p in _batch_inputs(case, seed):
            y = _f64(p.y)
            site0 = None if p.kind == "denoise" else _Deconv64(p.y.astype(np.float32), p.xi, p.kernel, 32)
            ep = _EP64(*p.shape, 1.0 / p.xi, y / p.xi, p.beta, site0=site0)
            ep.sweep(case["sweeps"], case["em"])
            post.append(ep.posterior())
        return dict(mean=torch.cat([m.reshape(-1) for m, _ in post]),
                    var=torch.cat([v.reshape(-1) for _, v in post]))
    elif kind == "cs":
        y, A, patterns = _cs_inputs(case, seed)
        A = _hadamard_rows(patterns, case["side"]) if A is None else A.double()
        y, xi, side = _f64(y), case["sigma"] ** 2, case["side"]
        ep = _EP64(side, side, 1.0 / xi, (A.T @ y).reshape(side, side) / xi, 1.0, site0=_cs64(A, y, xi))
    else:
        p = _warm_inputs(case, seed) if kind == "warm" else _deconv_inputs(case, seed)
        y = _f64(p.y)
        ep = _EP64(case["h"], case["w"], 1.0 / p.xi, y / p.xi, p.beta,
                   site0=_Deconv64(p.y.astype(np.float32), p.xi, p.kernel, case["probes"]))
        if kind == "warm":
            data = np.load(NET_FILE)
            layers = sum(1 for f in data.files if f[0] == "w" and f[1:].isdigit())
            params = [(_f64(data["w%d" % i]), _f64(data["b%d" % i])) for i in range(layers)]
            out = _net64(_features64(y[None], np.array([p.xi])), params)[0]
            ep.tau[:] = torch.clamp(torch.exp(out[1:]) / p.xi, min=1.0 / VAR_CAP)
            ep.nu[:] = ep.tau * (y + out[0])
    ep.sweep(case["sweeps"], case.get("em", 0))
    mean, var = ep.posterior()
    res = dict(mean=mean, var=var)
    if kind == "solve" or (case.get("em") and case["sweeps"] % case["em"] == 0):
        res["beta"] = float(ep.beta)
    return res
