"""Workloads for timing the RS-SRI-GF2 self-energy library through its public
entry points (paper_2005_12338_gb300.binding).

listed() names the workloads, draw() gives further ones of the same ranges,
prepare() makes what a user's program holds before the call (inputs on the
GPU, handles, output arrays), run() makes one pass through the entry points,
work() states what the pass cannot do without, and exact() evaluates the
method's equations (arXiv:2005.12338) in plain fp64 torch.

Kinds of workload:
  full    rssri_setup + rssri_sigma on a new problem: what a program does for
          every geometry or threshold it visits
  sample  rssri_sigma on a standing setup: more draws for a smaller error bar
  from_g  rssri_sigma_from_g: one iteration of a self-consistent loop, which
          brings its own dressed G(tau)
  batch   rssri_sigma_batch: several chains of uneven length, each set up
          before on its own stream
  train   rssri_cv_train: the learned control variate on an independent run
  energy  rssri_energy_static: Eq. 26 for a self-energy already in hand
Forms (arithmetic of the chain / of the deterministic block): "fp64"
(IEEE fp64 / IEEE fp64), "df64" (double-float / double-float), "sliced"
(double-float / sliced fp64-accurate on the tensor cores), "chosen" (bf16 /
sliced) and "tf32" (tf32 / sliced).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2005_12338_gb300 import binding

EPS_PRIME = 0.02  # the paper's screen of (ij|A)
BETA = 50.0
MU = 0.0
PREC = {"fp64": binding.RSSRI_PREC_FP64, "df64": binding.RSSRI_PREC_DF64,
        "sliced": binding.RSSRI_PREC_DF64, "chosen": binding.RSSRI_PREC_BF16,
        "tf32": binding.RSSRI_PREC_TF32}
ARITH = {"fp64": binding.RSSRI_DD_FP64, "df64": binding.RSSRI_DD_DF64,
         "sliced": binding.RSSRI_DD_OZ, "chosen": binding.RSSRI_DD_OZ,
         "tf32": binding.RSSRI_DD_OZ}


def _case(kind, n, n_aux, n_tau, n_s, eps, form, n_occ=None, cv=False, k=1):
    return dict(kind=kind, n=n, n_occ=n // 2 if n_occ is None else n_occ, n_aux=n_aux,
                n_tau=n_tau, n_s=n_s, eps=eps, form=form, cv=cv, k=k)


def listed():
    return [
        # the N = 20 correctness workload: the smallest problem anyone runs, in the default form
        dict(name="full_n20_fp64", **_case("full", 20, 60, 32, 64, 1e-2, "fp64")),
        # the paper's precision on the shortest chain of the 64-chain workload
        dict(name="full_n100_fp64", **_case("full", 100, 300, 32, 100, 1e-3, "fp64")),
        # fp64-accurate results without the tensor cores, between the two sizes the method is
        # run at, with fewer occupied than virtual orbitals
        dict(name="full_n150_df64", **_case("full", 150, 451, 24, 100, 1e-3, "df64", n_occ=63)),
        # the benchmark workload (N = 200, 64 tau points, 300 pairs) in the tensor-core form
        dict(name="full_n200_chosen", **_case("full", 200, 600, 64, 300, 1e-3, "chosen")),
        # a long chain of the 64-chain workload, few tau points
        dict(name="full_n500_chosen", **_case("full", 500, 1500, 4, 100, 1e-3, "chosen")),
        # more draws at the paper's threshold, where thousands of pairs are needed: fp64 ...
        dict(name="sample_n200_fp64", **_case("sample", 200, 600, 16, 64, 0.1, "fp64")),
        # ... and on the tensor cores
        dict(name="sample_n200_chosen", **_case("sample", 200, 600, 64, 300, 0.1, "chosen")),
        # the learned control variate on the tf32 chain, everything odd
        dict(name="sample_n131_tf32_cv",
             **_case("sample", 131, 393, 33, 151, 0.1, "tf32", n_occ=57, cv=True)),
        # one self-consistent iteration in the fp64-accurate tensor-core form
        dict(name="from_g_n120_sliced", **_case("from_g", 120, 360, 16, 64, 1e-2, "sliced")),
        # many systems: eight chains of N = 64 ... 256 enqueued together
        dict(name="batch_8_chosen", **_case("batch", 256, 768, 16, 64, 1e-3, "chosen", k=8)),
        # training the control variate on a short chain
        dict(name="train_n64", **_case("train", 64, 192, 16, 64, 0.1, "sliced")),
        # Eq. 26 alone, inside somebody else's loop
        dict(name="energy_n40", **_case("energy", 40, 1, 32, 1, 0.0, "fp64")),
    ]


# --------------------------------------------------------------- the ranges --
def _sizes(case):
    """(n, n_occ, n_aux) of every system of the case: one, or K chains of n/4 ... n."""
    if case["kind"] != "batch":
        return [(case["n"], case["n_occ"], case["n_aux"])]
    k, n = case["k"], case["n"]
    lo = max(24, n // 4)
    ns = [lo + round((n - lo) * i / max(1, k - 1)) for i in range(k)]
    return [(m, m // 2, 3 * m) for m in ns]


def _pairs(n, eps):
    """About how many pairs (i, j) keep a large part, for integrals decaying as exp(-|i-j|/3)."""
    h = min(n - 1, int(3.0 * math.log(0.7 / eps))) if eps > 0 else n - 1
    h = max(h, 0)
    return n * (2 * h + 1) - h * (h + 1)


def _block_flops(n, o, a, eps):
    """Flops of Sigma_DD at one tau point by the cheaper of two ways: over the kept pairs
    (exchange, then the dense products), or over (virtual, virtual, occupied) triples."""
    p = _pairs(n, eps)
    v = n - o
    return min(2.0 * a * p * p + 4.0 * a * n ** 3, 1.0 * n * n * v * v * o)


def _cost_ms(case):
    """A rough time of one pass, to keep drawn cases below the largest listed one."""
    tf = {"fp64": 1.0e9, "df64": 3.5e9, "sliced": 2.0e10, "chosen": 2.0e10, "tf32": 2.0e10}
    tc = {"fp64": 1.0e9, "df64": 3.5e9, "sliced": 3.5e9, "chosen": 1.0e11, "tf32": 5.0e10}
    ms, setup = 0.0, 0.0
    for n, o, a in _sizes(case):
        p = _pairs(n, case["eps"])
        rate = tf[case["form"]]
        block = (2.0 * a * p * p + 8.0 * a * n ** 3) / rate * case["n_tau"] + 0.3 * case["n_tau"]
        pre = block + (60.0 * a ** 3 + 2.0 * p * p * a) / min(rate, 3.5e9) + 5.0
        chain = 16.0 * n ** 3 * case["n_s"] * case["n_tau"] / tc[case["form"]]
        factors = 4.0 * case["n_s"] * (n * n + a) * a / min(rate, 3.5e9) + 2.0
        setup += pre
        ms += {"full": pre + chain + factors, "sample": chain + factors, "batch": chain + factors,
               "from_g": block + chain + factors, "train": 250.0 + chain + factors,
               "energy": 0.02}[case["kind"]]
    return ms, setup


def draw(rng):
    """One more case: sizes spread over their logarithm, odd ones among them."""
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    while True:
        kind = rng.choice(["full", "full", "full", "sample", "sample", "from_g", "batch",
                           "train", "energy"])
        if kind == "full":
            form = rng.choice(["fp64", "df64", "chosen", "sliced"])
            n = size(20, {"fp64": 140, "df64": 200, "chosen": 400, "sliced": 300}[form])
            case = _case(kind, n, 3 * n + rng.randint(-7, 7), size(2, 64), size(16, 300),
                         rng.choice([1e-3, 1e-2, 0.1]), form)
        elif kind == "sample":
            form = rng.choice(["fp64", "df64", "chosen", "tf32"])
            n = size(24, 220)
            case = _case(kind, n, 3 * n + rng.randint(-7, 7), size(4, 64), size(16, 400),
                         rng.choice([1e-2, 0.1]), form,
                         cv=form in ("chosen", "tf32") and rng.random() < 0.5)
        elif kind == "from_g":
            n = size(24, 144)
            case = _case(kind, n, 3 * n + rng.randint(-7, 7), size(2, 16), size(16, 128),
                         rng.choice([1e-3, 1e-2, 0.1]), rng.choice(["sliced", "df64", "fp64"]))
        elif kind == "batch":
            n = size(48, 256)
            case = _case(kind, n, 3 * n, size(4, 16), size(16, 64), rng.choice([1e-3, 1e-2]),
                         "chosen", k=rng.randint(3, 8))
        elif kind == "train":
            n = size(32, 80)
            case = _case(kind, n, 3 * n + rng.randint(-7, 7), size(8, 24), size(32, 96), 0.1,
                         "sliced")
        else:
            case = _case(kind, size(20, 200), 1, size(8, 64), 1, 0.0, "fp64")
        if kind not in ("batch", "energy"):
            case["n_occ"] = max(1, min(case["n"] - 1, int(case["n"] * rng.uniform(0.3, 0.55))))
        ms, setup = _cost_ms(case)
        if ms < 350.0 and setup < 600.0:
            return case


# --------------------------------------------------------------- the inputs --
def _tau_grid(n_tau):
    """Gauss-Legendre in ln(1 + tau/0.5) on (0, beta); the weights carry the Jacobian."""
    x, w = np.polynomial.legendre.leggauss(n_tau)
    umax = math.log1p(BETA / 0.5)
    tau = 0.5 * np.expm1(0.5 * (x + 1.0) * umax)
    return (torch.from_numpy(tau.copy()).cuda(),
            torch.from_numpy(0.5 * umax * w * (tau + 0.5)).cuda())


def _orbitals(n, gen):
    q, r = torch.linalg.qr(torch.randn((n, n), generator=gen, dtype=torch.float64,
                                       device="cuda").cpu())
    return (q * torch.sign(torch.diagonal(r))[None, :]).contiguous().cuda()


def _energies(n, n_occ, lo=-1.0, gap=0.2, hi=2.0):
    kw = dict(dtype=torch.float64, device="cuda")
    return torch.cat([torch.linspace(lo, -gap, n_occ, **kw),
                      torch.linspace(gap, hi, n - n_occ, **kw)]).contiguous()


def _system(n, n_occ, n_aux, n_tau, seed):
    """A hydrogen-chain-like problem: (ij|A) decaying over three sites, a well-conditioned
    metric, orthonormal orbitals with a 0.4 Eh gap."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    kw = dict(dtype=torch.float64, device="cuda")
    eri3 = torch.randn((n, n, n_aux), generator=gen, **kw)
    iu, ju = torch.triu_indices(n, n, 1, device="cuda")
    eri3[ju, iu, :] = eri3[iu, ju, :]
    idx = torch.arange(n, **kw)
    eri3 *= (torch.exp(-torch.abs(idx[:, None] - idx[None, :]) / 3.0)
             / math.sqrt(n_aux))[:, :, None]
    b = torch.randn((n_aux, n_aux), generator=gen, **kw)
    metric = b @ b.T / n_aux + 0.5 * torch.eye(n_aux, **kw)
    metric = (0.5 * (metric + metric.T)).contiguous()
    orb_c = _orbitals(n, gen)
    tau, tau_w = _tau_grid(n_tau)
    return eri3, metric, _energies(n, n_occ), orb_c, tau, tau_w


def _green(orb_e, orb_c, n_occ, tau):
    """Eq. 17 for non-interacting orbitals: G(tau) and G(beta - tau) for every tau."""
    co, cv = orb_c[:, :n_occ], orb_c[:, n_occ:]
    g = -torch.einsum("ia,ta,ja->tij", cv, torch.exp(-tau[:, None] * (orb_e[n_occ:] - MU)), cv)
    gb = -torch.einsum("ia,ta,ja->tij", co, torch.exp(tau[:, None] * (orb_e[:n_occ] - MU)), co)
    return g, gb


def _dressed(n, n_occ, orb_e, orb_c, tau, seed):
    """A dressed G of a self-consistent loop: nine tenths of it the quasiparticles, the rest
    satellites on rotated orbitals further from the gap; full rank, symmetric."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed) + 7919)
    g, gb = _green(orb_e, orb_c, n_occ, tau)
    g1, gb1 = _green(_energies(n, n_occ, -1.6, 0.35, 2.6), _orbitals(n, gen), n_occ, tau)
    g, gb = 0.9 * g + 0.1 * g1, 0.9 * gb + 0.1 * gb1
    return ((0.5 * (g + g.transpose(1, 2))).contiguous(),
            (0.5 * (gb + gb.transpose(1, 2))).contiguous())


def _net_params(seed):
    """Control-variate network parameters with an output of about 1 +- 0.1."""
    rng = np.random.default_rng(int(seed))
    sizes, parts = [10, 256, 256, 256, 1], []
    for k in range(4):
        w = rng.standard_normal((sizes[k + 1], sizes[k])) * np.sqrt(2.0 / sizes[k])
        parts += [(0.1 * w if k == 3 else w).ravel(), np.zeros(sizes[k + 1])]
    return np.concatenate(parts).astype(np.float32)


def _train_init(seed):
    """Hidden layers drawn, output layer zero: the network starts at c = 1."""
    p = _net_params(seed)
    p[-257:] = 0.0
    return p


def _options(case, seed):
    return binding.Handle.options(EPS_PRIME, case["eps"], case["n_s"], int(seed) % (1 << 31),
                                  precision=PREC[case["form"]], dd_arith=ARITH[case["form"]],
                                  cv=1 if case["cv"] else 0)


def prepare(case, seed):
    kind, nt, ns = case["kind"], case["n_tau"], case["n_s"]
    f64 = dict(dtype=torch.float64, device="cuda")
    if kind == "energy":
        gen = torch.Generator(device="cuda")
        gen.manual_seed(int(seed))
        n = case["n"]
        sig = torch.randn((nt, n, n), generator=gen, **f64)
        tau, tau_w = _tau_grid(nt)
        _, gb = _green(_energies(n, case["n_occ"]), _orbitals(n, gen), case["n_occ"], tau)
        return dict(case=case, sigma=(0.5 * (sig + sig.transpose(1, 2))).contiguous(),
                    gb=gb.contiguous(), tau_w=tau_w, e=torch.empty(1, **f64))
    opts = _options(case, seed)
    systems = [_system(n, o, a, nt, seed + 1000 * i) for i, (n, o, a) in enumerate(_sizes(case))]
    st = dict(case=case, opts=opts, arrays=systems,
              sigma=[torch.empty((nt, n, n), **f64) for n, _, _ in _sizes(case)],
              e_pair=[torch.empty(ns, **f64) for _ in systems])
    torch.cuda.synchronize()
    if kind == "batch":
        streams = [torch.cuda.Stream() for _ in systems]
        st["h"] = [binding.Handle(0, stream=s.cuda_stream) for s in streams]
        st["streams"] = streams
    else:
        st["h"] = [binding.Handle(0)]
    if kind == "train":
        st["init"] = _train_init(seed)
    if kind != "full":
        plain = _options(dict(case, cv=False), seed)
        for h, arrays, (n, o, a) in zip(st["h"], systems, _sizes(case)):
            h.setup(*arrays, n_occ=o, mu=MU, beta=BETA, opts=plain)
    if case["cv"]:
        st["h"][0].cv_set_params(_net_params(seed))
    if kind == "from_g":
        st["g"] = _dressed(case["n"], case["n_occ"], *systems[0][2:5], seed)
    return st


# ------------------------------------------------------------------ one pass --
def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind == "energy":
        s, gb, w, e = state["sigma"], state["gb"], state["tau_w"], state["e"]
        binding.check(binding.lib().rssri_energy_static(
            s.data_ptr(), gb.data_ptr(), w.data_ptr(), case["n"], case["n_tau"], case["n_occ"],
            e.data_ptr(), torch.cuda.current_stream().cuda_stream), "rssri_energy_static")
        return e
    opts, sig, ep = state["opts"], state["sigma"], state["e_pair"]
    if kind == "batch":
        e, se = binding.sigma_batch(state["h"], opts, sig, ep)
        return dict(sigma=sig, e_pair=ep, e_corr=e, e_stderr=se)
    h = state["h"][0]
    if kind == "train":
        before, after = h.cv_train(opts, state["init"], 100, 2048, 1e-3)
        return dict(loss_before=before, loss_after=after, params=h.export("CV_PARAMS"))
    if kind == "full":
        h.setup(*state["arrays"][0], n_occ=case["n_occ"], mu=MU, beta=BETA, opts=opts)
    g, gb = state["g"] if kind == "from_g" else (None, None)
    e, se, _ = h.sigma(opts, sig[0], ep[0], g=g, gb=gb)
    return dict(sigma=sig[0], e_pair=ep[0], e_corr=e, e_stderr=se)


def work(case):
    """Inputs read once, outputs written once; the flops of the cheapest known order of the
    products (2 n^3 per factor pair, sample pair and tau point for G given by its orbitals,
    8 n^3 for a general G)."""
    kind, nt, ns = case["kind"], case["n_tau"], case["n_s"]
    if kind == "energy":
        n = case["n"]
        return {"bytes": 16.0 * nt * n * n + 8.0 * nt, "flops": 2.0 * nt * n * n}
    by = fl = 0.0
    for n, o, a in _sizes(case):
        factors = 4.0 * ns * a * a + 4.0 * ns * a * (n * n + _pairs(n, case["eps"]))
        setup = 30.0 * a ** 3 + 2.0 * _pairs(n, case["eps"]) * a * a
        block = nt * _block_flops(n, o, a, case["eps"])
        chain = 2 * (8.0 if kind == "from_g" else 2.0) * ns * nt * n ** 3
        by += 8.0 * (n * n * a + nt * n * n + ns)  # (ij|A), Sigma, pair energies
        fl += chain + factors
        if kind == "full":
            by += 8.0 * (a * a + n * n)
            fl += setup + block
        elif kind == "from_g":
            by += 16.0 * nt * n * n
            fl += block
        elif kind == "train":
            fl += 100 * 6.0 * 2048 * (256 * 10 + 2 * 256 * 256 + 256)
    return {"bytes": by, "flops": fl}


# ------------------------------------------------- the equations in fp64 torch --
def _signs(seed, which, n_s, n_aux):
    """theta: -1 where bit 63 of the first SplitMix64 output (Steele, Lea and Flood, OOPSLA
    2014) from state seed XOR (which 2^60 + xi 2^20 + Q) is set, else +1."""
    xi = np.arange(n_s, dtype=np.uint64)[:, None] << np.uint64(20)
    c = (np.uint64(which) << np.uint64(60)) | xi | np.arange(n_aux, dtype=np.uint64)[None, :]
    z = (c ^ np.uint64(seed)) + np.uint64(0x9E3779B97F4A7C15)
    z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    z = z ^ (z >> np.uint64(31))
    return torch.from_numpy(1.0 - 2.0 * (z >> np.uint64(63)).astype(np.float64)).cuda()


def _block_orbital(k, orb_e, orb_c, o, tau):
    """Eq. 20 on v = sum_Q K^Q K^Q for the orbitals' G, summed over (a, b | c)."""
    n, _, a = k.shape
    co, cv = orb_c[:, :o], orb_c[:, o:]
    v = n - o
    b1 = torch.einsum("ipq,pa->iaq", k, cv)
    b2 = torch.einsum("ic,ibq->cbq", co, b1)
    ev = torch.exp(-tau[:, None] * (orb_e[o:] - MU))
    eo = torch.exp(tau[:, None] * (orb_e[:o] - MU))
    out = torch.zeros((len(tau), n, n), dtype=torch.float64, device="cuda")
    for c in range(o):
        vc = (b1.reshape(n * v, a) @ b2[c].T).reshape(n, v, v)
        mc = (2.0 * vc - vc.transpose(1, 2)).reshape(n, v * v)
        for t in range(len(tau)):
            # G(tau) G(tau) G(beta - tau): the product of three minus signs
            out[t] -= eo[t, c] * ((vc * ev[t][:, None] * ev[t]).reshape(n, v * v) @ mc.T)
    return out


def _block_general(k, g, gb):
    """The same for a general symmetric G(tau), over all pairs of orbital pairs."""
    n, _, a = k.shape
    kf = k.reshape(n * n, a)
    v = (kf @ kf.T).reshape(n, n, n, n).permute(0, 3, 1, 2).reshape(n * n, n * n).contiguous()
    out = torch.zeros_like(g)
    for t in range(g.shape[0]):
        pg = torch.einsum("ikq,km->imq", k, g[t])
        at = torch.einsum("kl,lmq->kmq", gb[t], pg).reshape(n * n, a)
        x = (v @ at).reshape(n, n, a)              # [m][j][Q] = sum_kl (mk|lj) At[k][l][Q]
        gam = kf.T @ at                            # Tr(K^Q' Gb K^Q G)
        u = 2.0 * (kf @ gam).reshape(n, n, a) - x
        out[t] = torch.einsum("imq,mjq->ij", pg, u)
    return out


def _net(params, x):
    p, off, sizes = torch.from_numpy(params.astype(np.float64)).cuda(), 0, [10, 256, 256, 256, 1]
    for i in range(4):
        w = p[off:off + sizes[i] * sizes[i + 1]].reshape(sizes[i + 1], sizes[i])
        off += w.numel()
        x = x @ w.T + p[off:off + sizes[i + 1]]
        off += sizes[i + 1]
        if i < 3:
            x = x / (1.0 + torch.exp(-x))
    return 1.0 + x[:, 0]


def _coefficients(params, sdd, g, gb, tau, k):
    """c_ij(tau) of the control-variate network from its ten features."""
    n = g.shape[1]
    i = torch.arange(n, device="cuda", dtype=torch.float64)
    one = torch.ones((n, n), dtype=torch.float64, device="cuda")
    r = k.pow(2).sum(dim=(1, 2)).sqrt()
    r = r / r.max()
    out = torch.empty_like(g)
    for t in range(g.shape[0]):
        dg, db = torch.diagonal(g[t]), torch.diagonal(gb[t])
        dg, db = dg / dg.abs().max(), db / db.abs().max()
        m = sdd[t].abs().max()
        f = [(i[:, None] - i[None, :]).abs() / n, one * (torch.log(tau[t]) / math.log(BETA)),
             sdd[t] / m if m > 0 else 0 * one, dg[:, None] * one, dg[None, :] * one,
             db[:, None] * one, db[None, :] * one, r[:, None] * one, r[None, :] * one,
             torch.eye(n, dtype=torch.float64, device="cuda")]
        out[t] = _net(params, torch.stack([x.reshape(-1) for x in f], 1)).reshape(n, n)
    return out


def _estimate(case, seed, arrays, sizes, g=None, gb=None, params=None):
    """Eqs. 7-16, 20, 25 and 26 for one system: (Sigma, pair energies, E_corr, stderr)."""
    eri3, metric, orb_e, orb_c, tau, tau_w = arrays
    n, o, a = sizes
    ns, nt = case["n_s"], case["n_tau"]
    lam, u = torch.linalg.eigh(metric)
    w = (u * lam ** -0.5) @ u.T
    m = eri3.abs().amax(dim=(0, 2))
    keep = eri3.abs() >= ((EPS_PRIME / n) * torch.minimum(m[:, None], m[None, :]))[:, :, None]
    k = (torch.where(keep, eri3, 0.0).reshape(n * n, a) @ w)
    k = torch.where(k.abs() >= case["eps"] * k.abs().max(), k, 0.0).reshape(n, n, a)
    del keep
    if g is None:
        g, gb = _green(orb_e, orb_c, o, tau)
        sdd = _block_orbital(k, orb_e, orb_c, o, tau)
    else:
        sdd = _block_general(k, g, gb)
    fac = []
    for which in (0, 1):
        th = _signs(int(seed) % (1 << 31), which, ns, a)
        fac.append(((th @ w) @ eri3.reshape(n * n, a).T).reshape(ns, n, n))
        fac.append((th @ k.reshape(n * n, a).T).reshape(ns, n, n))
    c = _coefficients(params, sdd, g, gb, tau, k) if params is not None else None
    sig = torch.empty_like(g)
    e_pair = torch.zeros(ns, dtype=torch.float64, device="cuda")
    for t in range(nt):
        f = []
        for x, y in ((fac[0], fac[2]), (fac[1], fac[3])):
            cm = x @ g[t] @ y
            bm = cm @ gb[t]
            tr = torch.diagonal(bm, dim1=1, dim2=2).sum(1)
            f.append(2.0 * tr[:, None, None] * cm - bm @ cm)
        ct = 1.0 if c is None else c[t]
        est = f[0] - ct * (f[1] - sdd[t])
        sig[t] = est.mean(0)
        e_pair -= tau_w[t] / (2.0 * o) * (est * gb[t].T).sum(dim=(1, 2))
    sig = 0.5 * (sig + sig.transpose(1, 2))
    return (sig, e_pair, float(e_pair.mean()), float(e_pair.std() / math.sqrt(ns)))


def exact(case, seed):
    kind = case["kind"]
    if kind == "train":
        return None  # a training run has no value in closed form
    if kind == "energy":
        s = prepare(case, seed)
        return -(s["tau_w"] * (s["sigma"] * s["gb"].transpose(1, 2)).sum(dim=(1, 2))).sum(
            0, keepdim=True) / (2.0 * case["n_occ"])
    tera = 0.0
    for n, o, a in _sizes(case):
        v = n - o
        block = 2.0 * n * n * v * v * o if kind != "from_g" else 2.0 * n ** 4 * a
        tera += (case["n_tau"] * block + 2.0 * n * v * v * o * a
                 + 16.0 * n ** 3 * case["n_s"] * case["n_tau"]) * 1e-12
    if tera > 14.0:
        return None  # fp64 runs at about 1 TFLOP/s
    got = []
    for i, sizes in enumerate(_sizes(case)):
        arrays = _system(*sizes, case["n_tau"], seed + 1000 * i)
        g = gb = None
        if kind == "from_g":
            g, gb = _dressed(sizes[0], sizes[1], *arrays[2:5], seed)
        got.append(_estimate(case, seed, arrays, sizes, g, gb,
                             _net_params(seed) if case["cv"] else None))
    out = dict(zip(("sigma", "e_pair", "e_corr", "e_stderr"), map(list, zip(*got))))
    return out if kind == "batch" else {k: v[0] for k, v in out.items()}
