"""GPU parity of the deconvolution path (prior sweep + CG/RBMC likelihood site)."""
import numpy as np
import pytest

from oracle import operators
from oracle.ep import EPOracle
from paper_2110_01585_gb300 import EPTV, OP_CONV_PERIODIC
from paper_2110_01585_gb300 import synthetic as syn

from ._cases import DECONV_CASES, oracle_run, probes, y32
from ._parity import assert_parity, cuda

pytestmark = pytest.mark.gpu


def _probes(S, n, seed):
    return syn.rbmc_probes(S, n, n, seed=seed)


def _gpu(p, sweeps, S, pr, em_every=0, cg_rtol=1e-9, **kw):
    torch = cuda()
    yt = torch.as_tensor(p.y.astype(np.float32), device="cuda")
    ep = EPTV(yt, p.xi, p.beta, op=OP_CONV_PERIODIC, kernel=p.kernel, rbmc_samples=S,
              cg_rtol=cg_rtol, **kw)
    ep.set_probes(torch.as_tensor(pr[0], dtype=torch.float32, device="cuda"),
                  torch.as_tensor(pr[1], dtype=torch.float32, device="cuda"))
    ep.sweep(sweeps, em_every=em_every)
    mu, var = ep.posterior()
    st = ep.status()
    out = mu.cpu().numpy(), var.cpu().numpy(), ep
    assert st == 0, st
    return out


@pytest.mark.parametrize("name", sorted(DECONV_CASES))
def test_deconv_parity(name):
    """Uniform 9x9 with EM, uniform 5x5 on a ragged 48x80 grid with EM, a
    non-separable 5x3 kernel, a 15x15 Gaussian (the first solve after one prior
    pass with capped prior sites needs thousands of iterations), and Algorithm 1
    as listed (likelihood site first: the first solve sees a flat cavity of
    precision 4e-8, the worst-conditioned system of the run)."""
    make, (S, seed), sweeps, em_every, order, opts = DECONV_CASES[name]
    p = make()
    pr = probes(p, S, seed)
    mu, var, ep = _gpu(p, sweeps, S, pr, em_every=em_every, **opts)
    mu_r, var_r = oracle_run(p, y32(p), pr, sweeps, em_every, order)
    assert_parity(mu, var, mu_r, var_r, p.y)
    ep.close()


@pytest.mark.parametrize("h,w", [(24, 400), (320, 24)])
def test_deconv_parity_512_point_transforms(h, w):
    """Padded sizes whose preconditioner rows (24 x 400, padded to 32 x 512) or
    columns (320 x 24, padded to 512 x 32) go through the register-resident
    512-point transforms; the oracle does every solve by FP64 CG on the FFT
    operator."""
    p = syn.deconv_problem(h, w, kernel=syn.uniform_kernel(5), bsnr_db=30.0, beta0=2.0, seed=31,
                           grf_length=8.0)
    S = 4
    pr = probes(p, S, 32)
    mu, var, ep = _gpu(p, 3, S, pr)
    o = EPOracle("deconv", y32(p), p.xi, p.beta, h, w, kernel=p.kernel, site0="rbmc_cg", probes=pr)
    o.run(3)
    mu_r, var_r = o.posterior()
    assert_parity(mu, var, mu_r, var_r, p.y)
    ep.close()


@pytest.mark.parametrize("h,w", [(24, 520), (520, 24)])
def test_deconv_parity_1024_point_transforms(h, w):
    """Padded sizes whose preconditioner rows (24 x 520, padded to 32 x 1024) or
    columns (520 x 24, padded to 1024 x 32) go through the register-resident
    1024-point transforms (one decimation-in-frequency step into two 512-point
    ones); the oracle does every solve by FP64 CG on the FFT operator."""
    p = syn.deconv_problem(h, w, kernel=syn.uniform_kernel(5), bsnr_db=30.0, beta0=2.0, seed=31,
                           grf_length=8.0)
    S = 4
    pr = probes(p, S, 32)
    mu, var, ep = _gpu(p, 3, S, pr)
    o = EPOracle("deconv", y32(p), p.xi, p.beta, h, w, kernel=p.kernel, site0="rbmc_cg", probes=pr)
    o.run(3)
    mu_r, var_r = o.posterior()
    assert_parity(mu, var, mu_r, var_r, p.y)
    ep.close()


def test_unit_kernel_equals_denoising_path():
    """H = I through the CG/RBMC route: diagonal precision, exact RB estimate."""
    torch = cuda()
    p = syn.denoise_problem(32, 64, sigma=0.1, beta=10.0, seed=11)
    p.kernel = np.ones((1, 1))
    pr = _probes(2, 32 * 64, 12)
    mu, var, ep = _gpu(p, 8, 2, pr)
    yt = torch.as_tensor(p.y.astype(np.float32), device="cuda")
    with EPTV(yt, p.xi, p.beta) as d:
        d.sweep(8)
        mu_d, var_d = (t.cpu().numpy() for t in d.posterior())
    np.testing.assert_allclose(mu, mu_d, rtol=1e-5, atol=1e-6)
    np.testing.assert_allclose(var, var_d, rtol=1e-5)
    ep.close()


def test_checkpoint_resume_deconv():
    torch = cuda()
    p = syn.deconv_problem(32, 32, kernel=syn.uniform_kernel(5), bsnr_db=30.0, seed=13,
                           grf_length=8.0)
    pr = _probes(4, 1024, 14)
    _, _, a = _gpu(p, 4, 4, pr, em_every=2)
    _, _, b = _gpu(p, 0, 4, pr, em_every=2)
    blob = a.state_export()
    a.sweep(4, em_every=2)
    b.state_import(blob)
    b.sweep(4, em_every=2)
    ma, va = a.posterior()
    mb, vb = b.posterior()
    assert torch.equal(ma, mb) and torch.equal(va, vb)
    a.close()
    b.close()


def test_library_probes_have_standard_normal_statistics():
    """The library's own SplitMix64/Box-Muller probes (no caller probes): run and
    check that the variance estimate is close to the exact-solve oracle."""
    torch = cuda()
    p = syn.deconv_problem(32, 32, kernel=syn.uniform_kernel(5), bsnr_db=30.0, seed=15,
                           grf_length=8.0)
    yt = torch.as_tensor(p.y.astype(np.float32), device="cuda")
    with EPTV(yt, p.xi, p.beta, op=OP_CONV_PERIODIC, kernel=p.kernel, rbmc_samples=64) as ep:
        ep.sweep(3)
        mu, var = (t.cpu().numpy() for t in ep.posterior())
    o = EPOracle("deconv", p.y, p.xi, p.beta, 32, 32, kernel=p.kernel, site0="exact")
    o.run(3)
    mu_r, var_r = o.posterior()
    # Monte Carlo error of the variance with 64 probes: a few percent at most
    assert np.median(np.abs(var / var_r - 1)) < 0.05
    assert np.max(np.abs(mu - mu_r)) < 0.05 * (p.y.max() - p.y.min())


def test_full_size_512_residual_and_site0_samples():
    """512^2, 9x9 uniform blur, BSNR 40 dB: after a sweep, the mean solve satisfies
    Q E = b everywhere (checked in FP64 with the oracle's operator), and the new
    likelihood site at sampled pixels follows the RB estimate and Eq. update_q0_x."""
    torch = cuda()
    h = w = 512
    S = 32
    p = syn.deconv_problem(h, w, kernel=syn.uniform_kernel(9), bsnr_db=40.0, beta0=1.0, seed=0)
    pr = _probes(S, h * w, 21)
    _, _, ep = _gpu(p, 2, S, pr, em_every=0)
    tau0, nu0 = (t.cpu().numpy().astype(np.float64) for t in ep.sites())
    ep.sweep(1)
    tau1, nu1 = (t.cpu().numpy().astype(np.float64) for t in ep.sites())
    blob = np.frombuffer(ep.state_export(), dtype=np.uint8)
    n = h * w
    off = 4 * 8 + 4 * 8 + 2 * 4 * 5 * n
    X = np.frombuffer(blob[off:].tobytes(), dtype=np.float64).reshape(1 + S, h, w)
    ep.close()
    d = tau1[1:].sum(axis=0)          # cavity precision of site 0 (prior sites of this sweep)
    ncav = nu1[1:].sum(axis=0)
    k = p.kernel
    def Q(v):
        return operators.conv_periodic_t(operators.conv_periodic(v, k), k) / p.xi + d * v
    b = operators.conv_periodic_t(p.y, k) / p.xi + ncav
    r = b - Q(X[0])
    assert np.linalg.norm(r) <= 1e-8 * np.linalg.norm(b)
    # probe systems
    g0 = float(np.sum(k * k)) / p.xi
    Ws = []
    for s in range(S):
        w_s = (operators.conv_periodic_t(pr[0][s].reshape(h, w), k) / np.sqrt(p.xi)
               + np.sqrt(d) * pr[1][s].reshape(h, w))
        rs = w_s - Q(X[s + 1])
        # probe solves stop at a relative residual of 1e-6 (mean solve: cg_rtol)
        assert np.linalg.norm(rs) <= 2e-6 * np.linalg.norm(w_s), s
        Ws.append(w_s)
    # site 0 at sampled pixels
    rng = np.random.default_rng(22)
    for rr, cc in rng.integers(0, 512, size=(50, 2)):
        qii = g0 + d[rr, cc]
        acc = 0.0
        for s in range(S):
            acc += (Ws[s][rr, cc] - qii * X[s + 1, rr, cc]) ** 2
        var = 1 / qii + acc / S / qii ** 2
        E = X[0, rr, cc]
        t_new = max(1 / var - d[rr, cc], 1e-8)
        n_new = t_new * E + d[rr, cc] * E - ncav[rr, cc]
        t_exp = 0.5 * t_new + 0.5 * tau0[0, rr, cc]
        n_exp = 0.5 * n_new + 0.5 * nu0[0, rr, cc]
        assert abs(tau1[0, rr, cc] / t_exp - 1) < 1e-4
        assert abs(nu1[0, rr, cc] - n_exp) <= 1e-4 * abs(t_exp) * (abs(E) + 0.1)


def test_config2_512_against_oracle_samples():
    """The deconvolution configuration at its stated size: 512 x 512, 9 x 9
    uniform periodic blur, BSNR 40 dB, 32 RBMC probes, beta0 = 1, six sweeps with
    the EM update after the fifth.  The FP64 oracle (every solve by CG to 1e-11)
    takes about 20 minutes for this on 8 cores, so its result is stored by
    tests/golden/make_deconv512.py (which calls only the oracle and the input
    generators) at 8192 sampled pixels, with the image-wide sums of the mean and
    the variance and the EM output."""
    import os

    from .golden import make_deconv512 as g

    ref = np.load(os.path.join(os.path.dirname(g.__file__), "deconv512_oracle.npz"))
    p, y32_, eps1, eps2 = g.inputs()
    # the same inputs as the stored run
    np.testing.assert_allclose(g.checksums(y32_, eps1, eps2), ref["checksums"], rtol=1e-12)
    torch = cuda()
    _, _, ep = _gpu(p, 0, g.S, (eps1, eps2))
    em = int(ref["em_every"])
    assert int(ref["sweeps"]) == em + 1
    ep.sweep(em, em_every=em)
    # ep_tv_em_beta recomputes N / a_u from the same (fifth) sweep: the beta the
    # in-sweep EM step just set, and the a_u it used
    beta, abar = ep.em_beta()
    ep.sweep(1)
    mu_t, var_t = ep.posterior()
    mu, var = (t.cpu().numpy().reshape(-1).astype(np.float64) for t in (mu_t, var_t))
    assert ep.status() == 0
    ep.close()
    assert abs(abar / float(ref["abar"]) - 1.0) < 1e-5, (abar, float(ref["abar"]))
    assert abs(beta / float(ref["beta"]) - 1.0) < 1e-5, (beta, float(ref["beta"]))
    idx = ref["idx"]
    assert_parity(mu[idx], var[idx], ref["mean"], ref["var"], p.y)
    assert abs(mu.sum() / float(ref["mean_sum"]) - 1.0) < 1e-5
    assert abs(var.sum() / float(ref["var_sum"]) - 1.0) < 1e-4


def test_deconv_mog2_prior_parity_and_no_em():
    """The MoG2-TV prior with the deconvolution likelihood site (Sec. II-B with
    Eq. tilted_P_1) against the oracle with the same probes, on an instance where
    thousands of site updates hit the variance cap; EM is refused for the mixture
    priors (Sec. IV defines it for l1-TV only)."""
    from paper_2110_01585_gb300 import PRIOR_MOG2, EPTVError

    from ._cases import MOG2_DECONV, mog2_deconv_problem, mog2_oracle_run
    c = MOG2_DECONV
    p = mog2_deconv_problem()
    pr = probes(p, c["S"], c["probe_seed"])
    theta = c["theta"]
    mu, var, ep = _gpu(p, c["sweeps"], c["S"], pr, prior=PRIOR_MOG2, omega=theta[0],
                       s1_sq=theta[1], s2_sq=theta[2])
    capped = ep.stats()["n_capped"]
    with pytest.raises(EPTVError):
        ep.sweep(1, em_every=1)
    with pytest.raises(EPTVError):
        ep.em_beta()
    ep.close()
    mu_r, var_r, capped_r = mog2_oracle_run(p, y32(p), pr)
    assert_parity(mu, var, mu_r, var_r, p.y)
    assert abs(capped - capped_r) <= max(4, 0.01 * capped_r), (capped, capped_r)


@pytest.mark.parametrize("h,w,periodic", [(60, 60, 1), (64, 128, 1), (33, 67, 0), (100, 250, 1), (131, 256, 0),
                                          (256, 40, 1), (300, 130, 1), (30, 511, 0), (520, 66, 1), (62, 1000, 1),
                                          (96, 96, 1), (192, 98, 1), (97, 191, 0), (384, 70, 1), (78, 350, 1)])
def test_deconv_parity_transform_sizes(h, w, periodic):
    """Every length of the preconditioner's warp transforms (64 to 512 points, powers of two
    and 3 2^k) along rows and columns, with 1024 and the shared-memory ones, with margins
    from none to nearly half the transform, even and odd; the oracle solves by FP64 CG."""
    p = syn.deconv_problem(h, w, kernel=syn.uniform_kernel(5), bsnr_db=30.0, beta0=2.0, seed=h + w,
                           grf_length=8.0)
    S = 3
    pr = probes(p, S, 52)
    mu, var, ep = _gpu(p, 2, S, pr, periodic=periodic)
    o = EPOracle("deconv", y32(p), p.xi, p.beta, h, w, kernel=p.kernel, site0="rbmc_cg", probes=pr,
                 periodic=bool(periodic))
    o.run(2)
    assert_parity(mu, var, *o.posterior(), p.y)
    ep.close()


@pytest.mark.parametrize("h,w,kernel,periodic", [(70, 66, 15, 1), (40, 100, 15, 1), (45, 67, 15, 0), (68, 70, 9, 1),
                                                 (72, 41, 9, 0), (66, 92, 5, 1), (34, 62, 3, 1)])
def test_deconv_parity_stencil_forms(h, w, kernel, periodic):
    """The paired stencil product for every halo, with rows of 4 k, even and odd lengths
    (float4, float2 and scalar staging) and tiles cut by the image's edges."""
    p = syn.deconv_problem(h, w, kernel=syn.uniform_kernel(kernel), bsnr_db=30.0, beta0=2.0, seed=h + w,
                           grf_length=8.0)
    S = 3
    pr = probes(p, S, 54)
    mu, var, ep = _gpu(p, 2, S, pr, periodic=periodic)
    o = EPOracle("deconv", y32(p), p.xi, p.beta, h, w, kernel=p.kernel, site0="rbmc_cg", probes=pr,
                 periodic=bool(periodic))
    o.run(2)
    assert_parity(mu, var, *o.posterior(), p.y)
    ep.close()


def _emulated_iterations(p, pr, d, ncav, rtol, torus, eta=3.2e-5):
    """Iterations of the first likelihood update (zero start): refinement passes of FP32 CG
    preconditioned by the windowed periodic extension into the torus, all
    systems in step, each pass down to max(eta |r|, rtol |b| / 2).  In FP32 as on the GPU:
    on these systems (flat regions have d near 1e-7) rounding costs CG iterations."""
    import scipy.fft as sf
    f4 = np.float32
    h, w = p.y.shape

    def axis(n, P):
        L = (P - n) // 2
        i = np.arange(P)
        src = np.where(i < n, i, np.where(i < n + L, i - n, np.where(i >= P - L, i - P + n, -1)))
        wgt = (src >= 0).astype(float)
        for k in range(-L, L):
            t = np.pi / 2 * (k + L + 0.5) / (2 * L)
            wgt[k % P] = np.sin(t)
            wgt[n + k] = np.cos(t)
        E = np.zeros((P, n))
        E[i[src >= 0], src[src >= 0]] = wgt[src >= 0]
        assert np.allclose(E.T @ E, np.eye(n))
        return E

    Er, Ec = axis(h, torus[0]), axis(w, torus[1])
    Er4, Ec4 = Er.astype(f4), Ec.astype(f4)
    k = p.kernel
    pad = np.zeros((Er.shape[0], Ec.shape[0]))
    pad[:k.shape[0], :k.shape[1]] = k
    filt = (1.0 / (np.abs(np.fft.fft2(pad)) ** 2 / p.xi + d.mean())).astype(f4)
    conv, conv_t = operators.conv_periodic, operators.conv_periodic_t
    d4 = d.astype(f4)
    gr, gc = (np.correlate(v, v, "full").astype(f4) for v in (k.sum(axis=1), k.sum(axis=0) / k.sum()))

    def stencil(v):
        out = v
        for ax, g in ((1, gc), (0, gr)):
            out = sum(g[i] * np.roll(out, i - len(g) // 2, axis=ax) for i in range(len(g)))
        return out

    def M(r):
        return Er4.T @ sf.ifft2(sf.fft2(Er4 @ r @ Ec4.T) * filt).real @ Ec4

    bs = [conv_t(p.y, k) / p.xi + ncav]
    for e1, e2 in zip(*pr):
        bs.append(conv_t(e1.reshape(h, w), k) / np.sqrt(p.xi) + np.sqrt(d) * e2.reshape(h, w))
    tols = [rtol] + [max(rtol, 1e-6)] * (len(bs) - 1)
    total = 0
    for b, tol in zip(bs, tols):
        r = b.astype(f4)
        nb = np.linalg.norm(b)
        stop, z, it = max(eta, 0.5 * tol) * nb, M(r), 0
        q, rz = z, np.sum(r * z, dtype=np.float64)
        while np.linalg.norm(r) > stop:
            aq = stencil(q) * f4(1.0 / p.xi) + d4 * q
            al = f4(rz / np.sum(q * aq, dtype=np.float64))
            r = r - al * aq
            z = M(r)
            rz, old = np.sum(r * z, dtype=np.float64), rz
            q = z + f4(rz / old) * q
            it += 1
        assert r.dtype == f4
        total = max(total, it)
    return total


@pytest.mark.parametrize("h,w,periodic,torus", [
    (76, 108, 1, (96, 128)), (45, 99, 0, (64, 128)), (40, 140, 1, (64, 192)), (128, 64, 1, (128, 64)),
    (24, 600, 1, (32, 1024)), (300, 90, 1, (384, 128)), (62, 62, 1, (96, 96))])
def test_preconditioner_iterations_are_those_of_the_windowed_extension(h, w, periodic, torus):
    """The preconditioner shows in the iteration count alone: the count of the first
    likelihood update is that of the emulation.  The target, 1e-4, is one that a single
    refinement pass meets (at 1e-9 the FP32 floor decides how many passes follow); FP32
    rounding moves a pass by an iteration or two."""
    p = syn.deconv_problem(h, w, kernel=syn.uniform_kernel(5), bsnr_db=30.0, beta0=2.0, seed=3, grf_length=8.0)
    p.y = p.y.astype(np.float32).astype(np.float64)
    S = 1
    pr = probes(p, S, 53)
    torch = cuda()
    # a stream of its own: the update runs as a graph, whose loop counts iterations one by
    # one (the host-driven loop launches them in fours)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        # sides that are not powers of two are solved to a quarter of cg_rtol
        rtol = 1e-4 if h & (h - 1) == 0 and w & (w - 1) == 0 else 4e-4
        _, _, ep = _gpu(p, 1, S, pr, periodic=periodic, cg_rtol=rtol, stream=stream)
        its = ep.stats()["cg_iters"]
        assert ep.solver_report()["passes"] == 1
        tau, nu = (t.cpu().numpy().astype(np.float64) for t in ep.sites())
        ep.close()
    ref = _emulated_iterations(p, pr, tau[1:].sum(axis=0), nu[1:].sum(axis=0), 1e-4, torus)
    assert abs(its - ref) <= 3 + 0.1 * ref, (its, ref)


@pytest.mark.parametrize("h,w", [(38, 68), (96, 96), (62, 62)])  # stencil, pointwise, paired stencil
@pytest.mark.parametrize("traced", [False, True])                # the graph, and the host-driven loop
def test_status_is_that_of_the_callers_target(h, w, traced):
    """Sides that are not powers of two aim at a quarter of cg_rtol or less; an iteration cap that
    ends a solve between the two raises no error, one that ends it before cg_rtol does."""
    torch = cuda()
    p = syn.deconv_problem(h, w, kernel=syn.uniform_kernel(5), bsnr_db=30.0, beta0=2.0, seed=h + w,
                           grf_length=8.0)
    y = torch.as_tensor(p.y.astype(np.float32), device="cuda")
    rtol, seen = 1e-3, set()
    for cap in range(1, 200):
        with EPTV(y, p.xi, p.beta, op=OP_CONV_PERIODIC, kernel=p.kernel, rbmc_samples=2, cg_rtol=rtol,
                  cg_max_iter=cap, stream=torch.cuda.Stream()) as ep:
            ep.trace(traced)
            ep.sweep(1)
            st, rep = ep.status(), ep.solver_report()
        worst = max(rep["relres_mean"], rep["relres_probe_max"])
        assert st == (5 if worst > rtol else 0), (cap, worst, st)
        seen.add("beyond" if worst > rtol else "between" if worst > 0.25 * rtol else "met")
        if worst <= 0.25 * rtol:
            break
    assert seen == {"beyond", "between", "met"}


@pytest.mark.parametrize("h,w", [(24, 1024), (1024, 24), (24, 2048), (2048, 24), (1300, 20), (20, 1300)])
def test_deconv_parity_long_transforms(h, w):
    """1024 points and the shared-memory transforms above, along rows and columns, with the
    axis filled (no copies, no window) and with a margin; the oracle solves by FP64 CG."""
    p = syn.deconv_problem(h, w, kernel=syn.uniform_kernel(5), bsnr_db=30.0, beta0=2.0, seed=h + w,
                           grf_length=8.0)
    S = 3
    pr = probes(p, S, 56)
    mu, var, ep = _gpu(p, 2, S, pr)
    o = EPOracle("deconv", y32(p), p.xi, p.beta, h, w, kernel=p.kernel, site0="rbmc_cg", probes=pr)
    o.run(2)
    assert_parity(mu, var, *o.posterior(), p.y)
    ep.close()


@pytest.mark.parametrize("h,w", [(62, 62), (38, 68), (96, 96), (192, 64)])  # with a window, and filling the torus
def test_probes_of_ragged_sizes_are_solved_to_an_eighth(h, w):
    """33 systems: a pass ends at half of the target, so the worst probe is between the last
    iteration's and that: 0.0625 of cg_rtol at an eighth (0.125 at a quarter, which let the
    variances be up to 1.4 times as far from exact ones), with some room for the true
    residual; the mean's target stays a quarter."""
    torch = cuda()
    p = syn.deconv_problem(h, w, kernel=syn.uniform_kernel(5), bsnr_db=30.0, beta0=2.0, seed=h + w,
                           grf_length=8.0)
    y = torch.as_tensor(p.y.astype(np.float32), device="cuda")
    with EPTV(y, p.xi, p.beta, op=OP_CONV_PERIODIC, kernel=p.kernel, rbmc_samples=32, cg_rtol=1e-3,
              cg_max_iter=10000) as ep:
        ep.sweep(1)
        rep = ep.solver_report()
        assert ep.status() == 0
    assert rep["relres_probe_max"] <= 0.08e-3 and rep["relres_mean"] <= 0.25e-3


def _torus(h, w, kh, kw):
    """The solver's choice of the preconditioner's torus (its rule, restated)."""
    lens = (64, 96, 128, 192, 256, 384, 512)

    def lengths(n):
        p2 = max(2, 1 << (n - 1).bit_length())
        return [p2] + [v for v in lens if n > 32 and n <= v <= 2 * n and v != p2]

    def its(P, n, k):
        x = (P - n) / max(k - 1, 1)
        return 1.0 if P == n else 1.0 + 0.2 * max(0.0, 3.0 - x) + 0.05 * max(0.0, 6.0 - x)

    def warp_cols(P, Q):
        return P in lens and Q % (256 * (12 if P % 3 == 0 else 16) // P) == 0

    return min((its(P, h, kh) * its(Q, w, kw) * (1.0 + P * Q / (3.0 * h * w)), i, (P, Q))
               for i, (P, Q) in enumerate((P, Q) for P in lengths(h) for Q in lengths(w))
               if not ((P % 3 == 0 or (Q % 3 == 0 and P in lens)) and not warp_cols(P, Q)))[2]


@pytest.mark.parametrize("h,w,periodic,torus", [(450, 40, 1, (512, 64)), (409, 35, 0, (512, 64)),
                                                (500, 66, 1, (512, 96)), (210, 40, 1, (256, 64)),
                                                (217, 35, 0, (256, 64)), (40, 216, 1, (64, 256)),
                                                (35, 470, 0, (64, 512))])
def test_deconv_parity_margins_of_256_and_512_points(h, w, periodic, torus):
    """Columns (and rows) of 256 and 512 points with a margin, whose gather and fold the sizes
    above leave out since 320 rows take 384 points: the torus is asserted, the results are
    the oracle's and the iterations those of the windowed extension on that torus."""
    assert _torus(h, w, 5, 5) == torus
    p = syn.deconv_problem(h, w, kernel=syn.uniform_kernel(5), bsnr_db=30.0, beta0=2.0, seed=h + w,
                           grf_length=8.0)
    S = 3
    pr = probes(p, S, 58)
    mu, var, ep = _gpu(p, 2, S, pr, periodic=periodic)
    o = EPOracle("deconv", y32(p), p.xi, p.beta, h, w, kernel=p.kernel, site0="rbmc_cg", probes=pr,
                 periodic=bool(periodic))
    o.run(2)
    assert_parity(mu, var, *o.posterior(), p.y)
    ep.close()
    test_preconditioner_iterations_are_those_of_the_windowed_extension(h, w, periodic, torus)


@pytest.mark.parametrize("kernel", ["nonseparable 5x3", "separable 3x7"])
@pytest.mark.parametrize("h,w,S", [(64, 64, 2), (64, 64, 3),    # a pass as one kernel
                                   (64, 128, 3), (96, 96, 2),   # three kernels per iteration
                                   (32, 64, 2)])                # columns in shared memory
def test_deconv_parity_pointwise_products_of_any_blur(h, w, S, kernel):
    """Images that fill the torus form Q z from the transform of the kernel, whatever its form;
    the true residual that ends a solve comes from the taps.  Rectangular kernels, separable
    and not, with even and odd numbers of systems, against the oracle."""
    if kernel == "nonseparable 5x3":
        k = np.random.default_rng(4).random((5, 3)) ** 2
        assert np.linalg.matrix_rank(k) == 3
    else:
        k = np.outer([1.0, 2.0, 1.5], [1.0, 2.0, 3.0, 4.0, 3.5, 2.0, 0.5])
    assert _torus(h, w, *k.shape) == (h, w)
    p = syn.deconv_problem(h, w, kernel=k / k.sum(), bsnr_db=30.0, beta0=2.0, seed=h + w, grf_length=8.0)
    pr = probes(p, S, 60)
    mu, var, ep = _gpu(p, 3, S, pr)
    rep = ep.solver_report()
    assert rep["relres_mean"] <= 1e-9 and rep["relres_probe_max"] <= 1e-6
    o = EPOracle("deconv", y32(p), p.xi, p.beta, h, w, kernel=p.kernel, site0="rbmc_cg", probes=pr)
    o.run(3)
    assert_parity(mu, var, *o.posterior(), p.y)
    ep.close()
