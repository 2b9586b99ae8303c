"""What is measured: the work a spectral-function run has this library do, each case one call (or
one short sequence of calls) through the package's public entry points, at the sizes of the
repository's own workloads (synth.WORKLOADS, the 6 x 6 symmetry projection, the 300-state Krylov
step) and, drawn, at others of the same ranges: chains of 12 to 96 sites and lattices of 4 x 4 to
16 x 16, odd and ragged hidden widths and walker counts, float64, float32 and mixed contexts.

A case is {"kind", "prec", "Lx", "Ly", "M", "B", ...}.  The kinds:

  iteration    one natural-gradient iteration (sweep, local target, update, theta refresh), the
               inner loop of every projection step, through batch_run
  scan         the same for several sequences at once (a momentum scan), captured in one CUDA
               graph and replayed, as batch.Batch runs them
  sweep        mc_sweep: the Metropolis sweep alone
  target       cheb_local_target: R = phi_n / psi_n of a step n >= 2
  solve        sr_step: estimators, force and the shifted solve (matrix-free CG or explicit S)
  grad         the differentiable log psi, forward and backward (overlap loss)
  sym          sym_hbtilde: the momentum projection of stored states
  krylov       cheb_gram and cheb_krylov over the stored states
  extrapolate  cheb_extrapolate: linear prediction of higher moments

Parameters are random complex RBMs of the workloads' scale (the fitted one a little away from the
two it recurses from), walkers random S^z = 0 configurations; theta, log psi and tanh theta that a
call takes are formed here in 64 bits and rounded.  R of a solve is the ratio of a nearby RBM's
amplitude to psi with a scatter of 30% that no RBM holds, what a fit sees of phi_n / psi_n.
"""

import math

import numpy as np
import torch

from paper_2103_08804_gb300 import api, autograd, driver, synth

PREC = {"fp64": api.FP64, "fp32": api.FP32, "mixed": api.MIXED}
WP = 0.9875
Q = {"1d": (math.pi / 2, 0.0), "2d": (math.pi, 0.0)}


def _case(name, kind, prec, Lx, Ly, M, B, **kw):
    return {"name": name, "kind": kind, "prec": prec, "Lx": Lx, "Ly": Ly, "M": M, "B": B, **kw}


def listed():
    return [
        # the smallest system: a 12-site chain in float64 with the direct solve; launches and
        # short serial chains count
        _case("chain12_iteration", "iteration", "fp64", 12, 1, 12, 1024, sigma=0.05, shift=1e-3,
              solver="cholesky"),
        # the 16 x 16 lattice, the largest matrix-free workload: the whole iteration, then its parts
        _case("square16_iteration", "iteration", "mixed", 16, 16, 256, 65536, sigma=0.01,
              shift=0.1, solver="cg"),
        _case("square16_sweep", "sweep", "mixed", 16, 16, 256, 65536, sigma=0.01, sweeps=1),
        _case("square16_target", "target", "mixed", 16, 16, 256, 65536, sigma=0.01),
        _case("square16_solve", "solve", "mixed", 16, 16, 256, 65536, sigma=0.01, shift=0.1,
              solver="cg"),
        # the 64-site chain in plain float32: the update with the CG on the float32 pipes
        _case("chain64_solve_fp32", "solve", "fp32", 64, 1, 128, 16384, sigma=0.02, shift=1e-3,
              solver="cg"),
        # the 10 x 10 lattice: explicit S (P = 10,200) and the direct solve
        _case("square10_solve_explicit", "solve", "mixed", 10, 10, 100, 32768, sigma=0.01,
              shift=1e-2, solver="cholesky"),
        # a momentum scan: two momenta of the 8 x 8 lattice and two chains side by side
        _case("scan", "scan", "mixed", 8, 8, 128, 8192, sigma=0.02, shift=0.1, solver="cg",
              chain_a=48, chain_b=96, ctas=38),
        # training outside the natural gradient: log psi with its gradient at the 10 x 10 size
        _case("square10_grad", "grad", "fp32", 10, 10, 100, 32768, sigma=0.01),
        # symmetry projection of the 6 x 6 lattice, six of its stored states
        _case("sym6", "sym", "fp32", 6, 6, 72, 4096, sigma=0.02, states=6),
        # the Krylov step of a finished sequence: 300 states at 65536 samples
        _case("krylov300", "krylov", "mixed", 16, 16, 256, 65536, states=300),
        # moments of every momentum of the 6 x 6 lattice continued from 300 to 3000
        _case("extrapolate36", "extrapolate", "fp64", 6, 6, 72, 64, sequences=36, known=300,
              order=100, out=3000),
    ]


def _spread(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _lattice(rng, max_n=256):
    while True:
        if rng.random() < 0.5:
            Lx, Ly = 2 * rng.randint(6, 48), 1
        else:
            Lx, Ly = rng.randint(4, 16), rng.randint(4, 16)
        if Lx * Ly % 2 == 0 and Lx * Ly <= max_n:
            return Lx, Ly


def draw(rng):
    kind = rng.choice(["iteration", "scan", "sweep", "target", "solve", "solve", "solve", "grad",
                       "sym", "krylov", "extrapolate"])
    prec = rng.choice(["fp32", "mixed", "mixed"])
    Lx, Ly = _lattice(rng)
    M, B = _spread(rng, 12, 256), _spread(rng, 512, 65536)
    sigma = rng.uniform(0.01, 0.03)
    if kind in ("iteration", "sweep", "target"):
        if rng.random() < 0.15:  # float64 runs are small
            prec, M, B = "fp64", min(M, 64), min(B, 2048)
            Lx, Ly = _lattice(rng, 36)
        c = _case("", kind, prec, Lx, Ly, M, B, sigma=sigma)
        if kind == "sweep":
            c["sweeps"] = rng.choice([1, 1, 2, 4]) if Lx * Ly * M * B < 1 << 28 else 1
        if kind == "iteration":
            c.update(shift=0.1 if prec != "fp64" else 1e-3, solver="cg" if prec != "fp64" else "cholesky")
            if prec == "fp64":
                c["M"] = min(M, 16)
    elif kind == "scan":
        c = _case("", kind, "mixed", 8, 8, _spread(rng, 64, 128), _spread(rng, 1024, 8192),
                  sigma=sigma, shift=0.1, solver="cg", chain_a=2 * rng.randint(12, 32),
                  chain_b=2 * rng.randint(32, 48), ctas=rng.choice([19, 38, 76]))
    elif kind == "solve":
        if rng.random() < 0.4:  # explicit S: P below about 10,000
            Lx, Ly = _lattice(rng, 100)
            M = min(M, max(12, 10000 // (Lx * Ly)))
            B = _spread(rng, 1024, 32768)
            c = _case("", kind, prec, Lx, Ly, M, B, sigma=sigma, shift=1e-2, solver="cholesky")
            if prec == "fp32":  # S is accumulated in float64 there: smaller systems
                c["M"], c["B"] = min(M, max(12, 2000 // (Lx * Ly))), min(B, 4096)
        else:
            c = _case("", kind, prec, Lx, Ly, M, B, sigma=sigma, shift=0.1, solver="cg")
            if prec == "fp32":
                c["B"] = min(B, 16384)
    elif kind == "grad":
        c = _case("", kind, prec, Lx, Ly, M, B, sigma=sigma)
    elif kind == "sym":
        L = rng.choice([4, 6, 6, 8])
        c = _case("", kind, "fp32", L, L, _spread(rng, 12, 128), _spread(rng, 64, 4096 * 16 // (L * L)),
                  sigma=sigma, states=rng.randint(1, 5))
    elif kind == "krylov":
        Nm = _spread(rng, 12, 300)
        c = _case("", kind, "mixed", 8, 8, 64, _spread(rng, max(2048, 8 * Nm), 65536), states=Nm)
    else:
        known = rng.randint(80, 300)
        c = _case("", kind, "fp64", 6, 6, 72, 64, sequences=rng.randint(1, 36), known=known,
                  order=rng.randint(10, known // 3), out=known * rng.randint(2, 10))
    del c["name"]
    return c


# ------------------------------------------------------------------ inputs

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _rbm(seed, N, M, sigma):
    """Random complex RBM, complex128 on the GPU (the same values for every precision)."""
    return torch.from_numpy(synth.rbm_params(seed, N, M, sigma)).cuda()


def _sz0(seed, B, N):
    """Random S^z = 0 configurations, int8 [B, N]."""
    r = torch.rand(B, N, device="cuda", generator=_gen(seed))
    top = r.argsort(dim=1)[:, : N // 2]
    s = torch.full((B, N), -1, dtype=torch.int8, device="cuda")
    return s.scatter_(1, top, 1)


def _cd(case):
    return torch.complex128 if case["prec"] == "fp64" else torch.complex64


def _theta64(p, s, N, M):
    """theta = b + sigma W in 64 bits."""
    sd = s.double()
    W = p[N + M:].reshape(N, M)
    return torch.complex(sd @ W.real.contiguous(), sd @ W.imag.contiguous()) + p[N:N + M]


def _logpsi64(p, s, N, M, th=None):
    th = _theta64(p, s, N, M) if th is None else th
    sg = torch.where(th.real < 0, -1.0, 1.0)
    z = th * sg
    v = (z + torch.log(1.0 + torch.exp(-2.0 * z))).sum(1)
    sd = s.double()
    return v + torch.complex(sd @ p[:N].real.contiguous(), sd @ p[:N].imag.contiguous())


def _inputs(case, seed, Lx=None, Ly=None, M=None):
    """Parameters (64-bit values of the context's precision), walkers, and what goes with them."""
    Lx, Ly, M = Lx or case["Lx"], Ly or case["Ly"], M or case["M"]
    N, sg, cd = Lx * Ly, case["sigma"], _cd(case)

    def rnd(x):
        return x.to(cd).to(torch.complex128)

    psi = rnd(_rbm(1000 * seed + 1, N, M, sg))
    x = {"N": N, "M": M, "Lx": Lx, "Ly": Ly, "cd": cd, "prev2": psi}
    x["prev"] = rnd(psi + _rbm(1000 * seed + 2, N, M, 0.3 * sg))
    x["cur"] = rnd(x["prev"] + _rbm(1000 * seed + 3, N, M, 0.1 * sg))
    x["tgt"] = rnd(x["cur"] + _rbm(1000 * seed + 4, N, M, 0.3 * sg))
    x["spins"] = _sz0(1000 * seed + 5, case["B"], N)
    x["E0"], x["a"] = synth.safe_rescaling(Lx, Ly)
    x["beta"] = torch.tensor([0.7 + 0.1j, 0.9 - 0.05j], dtype=torch.complex128, device="cuda")
    x["q"] = Q["1d" if Ly == 1 else "2d"]
    return x


def _at_walkers(x):
    """theta, log psi, tanh theta of the current RBM at the walkers (64 bits, then rounded)."""
    th = _theta64(x["cur"], x["spins"], x["N"], x["M"])
    lp = _logpsi64(x["cur"], x["spins"], x["N"], x["M"], th)
    return th.to(x["cd"]), lp.to(x["cd"]), torch.tanh(th).to(x["cd"])


def _ctx(case, x, stream=None, B=None):
    return api.Context(x["Lx"], x["Ly"], x["M"], B or case["B"], prec=PREC[case["prec"]],
                       explicit_s=case.get("solver") == "cholesky", stream=stream)


def _solver(case):
    return api.SOLVE_CHOLESKY if case["solver"] == "cholesky" else api.SOLVE_CG


def _sequence(case, seed, stream, Lx=None, Ly=None, M=None):
    """A driver.Sequence in the middle of projection step n = 3, its fixed buffers filled."""
    x = _inputs(case, seed, Lx, Ly, M)
    theta, lp, _ = _at_walkers(x)
    ctx = _ctx(case, x, stream)
    cfg = driver.SeqConfig(Lx=x["Lx"], Ly=x["Ly"], M=x["M"], q=x["q"], n_moments=4, n_iter=1,
                           shift=case["shift"], dgamma=0.5, E0=x["E0"], a=x["a"], Wp=WP,
                           seed=seed, solver=_solver(case), cg_maxit=50, cg_tol=1e-4, krylov=False)
    host = x["spins"].cpu().numpy()
    seq = driver.Sequence(ctx, cfg, x["prev2"].cpu().numpy(), host, host[:1], graphs=True)
    seq.prev_buf.copy_(x["prev"])
    seq.prev2_buf.copy_(x["prev2"])
    seq.beta_buf.copy_(x["beta"].flip(0))
    # the recorded state that every pass starts from
    at = {"work": x["cur"].to(x["cd"]), "spins": x["spins"], "theta": theta, "lp": lp}
    return seq, at


def _restore(seq, at):
    for k, v in at.items():
        getattr(seq, k).copy_(v)


def _result(seq):
    return {"params": seq.work, "spins": seq.spins, "tanh": seq.tanh, "R": seq.R,
            "theta": seq.theta, "logpsi": seq.lp}


def _columns(case, seed):
    """Columns B_n(s), (H' t_n)(s)/psi(s) of states t_n = T_n(x) t_0 over D levels x in (-1, 1),
    each with its own fit error of 3%, seen through an isometry onto the samples."""
    Nm, B = case["states"], case["B"]
    D = min(1024, B // 2)
    g = _gen(1000 * seed + 6)
    x = torch.cos(math.pi * (torch.arange(D, device="cuda", dtype=torch.float64) + 0.5) / D) * 0.95
    t0 = torch.exp(-2.0 * (x - 0.2) ** 2)
    t0 = t0 / t0.norm()
    n = torch.arange(Nm, device="cuda", dtype=torch.float64)
    t = torch.cos(n[:, None] * torch.acos(x)[None, :]) * t0
    t = t.to(torch.complex64)
    t[1:] += 0.03 / math.sqrt(D) * torch.randn(Nm - 1, D, dtype=torch.complex64, device="cuda", generator=g)
    t = t * torch.exp(2j * math.pi * torch.rand(D, device="cuda", generator=g)).to(torch.complex64)
    pos = torch.randperm(B, device="cuda", generator=g)[:D]

    def spread(v):
        full = torch.zeros(Nm, B, dtype=torch.complex64, device="cuda")
        full[:, pos] = v
        return torch.fft.fft(full).contiguous()

    return spread(t), spread(t * x.to(torch.complex64))


def _moments(case, seed):
    """Moments of damped poles inside the band with sampling noise of 1e-3 mu_0."""
    r = np.random.default_rng(1000 * seed + 7)
    out = []
    for _ in range(case["sequences"]):
        K = 24
        x, w = r.uniform(-0.9, 0.9, K), r.uniform(0.1, 1.0, K)
        n = np.arange(case["known"])
        mu = (w[:, None] * np.cos(np.arccos(x)[:, None] * n) * np.exp(-0.01 * n)).sum(0) / w.sum()
        out.append(mu + 1e-3 * (r.standard_normal(len(n)) + 1j * r.standard_normal(len(n))))
    return torch.from_numpy(np.array(out)).cuda()


REG = 1e-6  # Tikhonov term at the square of the moments' noise


def prepare(case, seed):
    kind, s = case["kind"], {"kind": case["kind"]}
    if kind == "krylov":
        Nm = case["states"]
        s["Bm"], s["HBm"] = _columns(case, seed)
        s["ctx"] = api.Context(case["Lx"], case["Ly"], case["M"], 64, prec=PREC[case["prec"]])
        s["G"] = torch.empty(Nm, Nm, dtype=torch.complex128, device="cuda")
        s["H"] = torch.empty_like(s["G"])
        s["mu"] = torch.zeros(2 * Nm, dtype=torch.complex128, device="cuda")
        s["poles"] = torch.zeros(Nm, dtype=torch.float64, device="cuda")
        s["weights"] = torch.zeros_like(s["poles"])
        s["rank"] = torch.zeros(1, dtype=torch.int32, device="cuda")
        return s
    if kind == "extrapolate":
        s["mu"] = _moments(case, seed)
        s["ctx"] = api.Context(case["Lx"], case["Ly"], case["M"], 64, prec=api.FP64)
        s["args"] = (case["order"], case["known"] // 2, case["out"], REG)
        return s
    if kind == "iteration":
        s["seq"], s["at"] = _sequence(case, seed, torch.cuda.current_stream())
        s["desc"] = s["seq"].iter_desc(3)
        return s
    if kind == "scan":
        shapes = [(case["Lx"], case["Ly"], case["M"])] * 2
        shapes += [(n, 1, 2 * n) for n in (case["chain_a"], case["chain_b"])]
        s["seqs"], s["at"], descs = [], [], []
        for k, (Lx, Ly, M) in enumerate(shapes):
            seq, at = _sequence(case, 10 * seed + k, torch.cuda.Stream(), Lx, Ly, M)
            if seq.ctx.fused_cg():
                seq.ctx.set_fcg_ctas(case["ctas"])
            _restore(seq, at)
            s["seqs"].append(seq)
            s["at"].append(at)
            descs.append(seq.iter_desc(3))
        main = torch.cuda.current_stream()
        api.batch_run(descs, 1, main)  # loads every kernel, as Batch does before it captures
        torch.cuda.synchronize()
        s["graph"], cap = torch.cuda.CUDAGraph(), torch.cuda.Stream()
        cap.wait_stream(main)
        with torch.cuda.graph(s["graph"], stream=cap):
            api.batch_run(descs, 1, cap)
        main.wait_stream(cap)
        for seq in s["seqs"]:
            seq.ctr.zero_()  # the walkers' random streams start here
        return s
    x = _inputs(case, seed)
    s["ctx"], s["spins"] = _ctx(case, x), x["spins"]
    if kind == "sym":
        s["params"] = torch.stack([_rbm(1000 * seed + 10 + n, x["N"], x["M"], case["sigma"])
                                   for n in range(case["states"])]).to(x["cd"])
        s["lp"] = _logpsi64(x["prev2"], x["spins"], x["N"], x["M"]).to(x["cd"])
        s["hp"] = (x["E0"], x["a"], WP)
        return s
    theta, lp, T = _at_walkers(x)
    s.update(theta=theta, lp=lp, tanh=T, params=x["cur"].to(x["cd"]))
    B = case["B"]
    if kind == "sweep":
        s["rng"], s["sweeps"] = api.Philox(seed, 0), case["sweeps"]
        s["acc"] = torch.zeros(B, dtype=torch.int32, device="cuda")
    elif kind == "target":
        s["prev"], s["prev2"] = x["prev"].to(x["cd"]), x["prev2"].to(x["cd"])
        s["x"] = x
        s["R"] = torch.empty(B, dtype=x["cd"], device="cuda")
    else:
        R = 0.8 * torch.exp(_logpsi64(x["tgt"], x["spins"], x["N"], x["M"]) -
                            _logpsi64(x["cur"], x["spins"], x["N"], x["M"]))
        R = R * (1 + 0.3 * torch.randn(B, dtype=torch.complex128, device="cuda",
                                       generator=_gen(1000 * seed + 8)))
        s["R"] = R.to(x["cd"])
        if kind == "solve":
            s["opts"] = dict(dgamma=0.5, shift=case["shift"], solver=_solver(case), cg_maxit=50,
                             cg_tol=1e-4)
        else:
            s["leaf"] = s["params"].clone().requires_grad_(True)
            s["lp0"] = _logpsi64(x["prev"], x["spins"], x["N"], x["M"]).to(x["cd"])
    return s


def run(state):
    kind, c = state["kind"], state.get("ctx")
    if kind == "iteration":
        _restore(state["seq"], state["at"])
        api.batch_run([state["desc"]], 1, torch.cuda.current_stream())
        return _result(state["seq"])
    if kind == "scan":
        for seq, at in zip(state["seqs"], state["at"]):
            _restore(seq, at)
        state["graph"].replay()
        return [_result(seq) for seq in state["seqs"]]
    if kind == "sweep":
        c.mc_sweep(state["params"], state["spins"], state["theta"], state["sweeps"], state["rng"],
                   logpsi_out=state["lp"], tanh_out=state["tanh"], n_accepted=state["acc"])
        return {k: state[k] for k in ("spins", "theta", "lp", "tanh", "acc")}
    if kind == "target":
        x = state["x"]
        b = x["beta"]
        return c.cheb_local_target(3, c.state(state["prev"]), c.state(state["prev2"]), b[1:2], b[0:1],
                                   x["E0"], x["a"], WP, state["spins"], state["lp"], state["R"])
    if kind == "solve":
        p = state["params"].clone()
        c.sr_step(p, state["spins"], state["tanh"], state["R"], **state["opts"])
        return p
    if kind == "grad":
        leaf = state["leaf"]
        leaf.grad = None
        loss = autograd.overlap_loss(c, leaf, state["spins"], state["lp0"], state["R"])
        loss.backward()
        return {"loss": loss.detach(), "grad": leaf.grad}
    if kind == "sym":
        return list(c.sym_hbtilde(state["params"], state["spins"], state["lp"], state["hp"]))
    if kind == "krylov":
        c.cheb_gram(state["Bm"], state["HBm"], state["G"], state["H"])
        c.cheb_krylov(state["G"], state["H"], 1e-10, len(state["mu"]), state["mu"], state["poles"],
                      state["weights"], state["rank"])
        return {k: state[k] for k in ("G", "H", "mu", "poles", "weights", "rank")}
    order, n0, n_out, reg = state["args"]
    return c.cheb_extrapolate(state["mu"], order, n0, n_out, reg=reg)


# -------------------------------------------------------------------- work

CG_ITS = 16  # CG iterations a solve to 1e-4 needs at least at shift 0.1 (at most 50 are allowed)


def _work_iteration(case, N, Nb, M, B, parts):
    """Bytes and flops of the parts of an iteration.  An antiparallel exchange costs 14 flops per
    hidden unit (a complex multiply-add and a complex multiply), half the bonds are antiparallel."""
    cs = 16 if case["prec"] == "fp64" else 8
    P = N + M + N * M
    by, fl = 0.0, 0.0
    if "sweep" in parts:
        n = case.get("sweeps", 1)
        by += 2 * B * N + cs * B * (3 * M + 1) + cs * P
        fl += 14.0 * n * B * (N / 2) * M
    if "target" in parts:
        by += B * N + 2 * cs * B + 2 * cs * P
        fl += B * (14.0 * (Nb / 2) * M + 8.0 * N * M)
    if "solve" in parts:
        by += B * (N + cs * M + cs) + 2 * cs * P
        fl += 8.0 * B * N * M  # the two sums of the estimators
        if case["solver"] == "cg":
            fl += CG_ITS * 8.0 * B * N * M
        else:
            # S from the products sigma_i sigma_i' and conj(T_j) T_j', then P^3 / 3 complex
            fl += 1.0 * B * N * N * M * M + 8.0 * P ** 3 / 3
    if "theta" in parts:
        by += B * (N + cs * M + cs) + cs * P
        fl += 4.0 * B * N * M
    return by, fl


def work(case):
    kind, M, B = case["kind"], case["M"], case["B"]
    N = case["Lx"] * case["Ly"]
    Nb = N if case["Ly"] == 1 else 2 * N
    P = N + M + N * M
    if kind in ("iteration", "sweep", "target", "solve"):
        parts = {"iteration": ("sweep", "target", "solve", "theta")}.get(kind, (kind,))
        by, fl = _work_iteration(case, N, Nb, M, B, parts)
    elif kind == "scan":
        by = fl = 0.0
        shapes = [(N, Nb, M)] * 2 + [(n, n, 2 * n) for n in (case["chain_a"], case["chain_b"])]
        for n, nb, m in shapes:
            b, f = _work_iteration(case, n, nb, m, B, ("sweep", "target", "solve", "theta"))
            by, fl = by + b, fl + f
    elif kind == "grad":
        by, fl = 2 * B * N + 24 * B + 16 * P, 8.0 * B * N * M
    elif kind == "sym":
        S, conf = case["states"], 4 * N * B
        by = B * N + 8 * S * (P + 2 * N * B)
        fl = S * conf * (4.0 * N * M + 14.0 * (Nb / 2) * M)
    elif kind == "krylov":
        S = case["states"]
        # two Gram matrices, two complex Hermitian eigenproblems (about 9 n^3 complex), 2 S steps
        by = 16 * S * B + 6 * 16 * S * S
        fl = 2 * 4.0 * S * S * B + 2 * 36.0 * S ** 3 + 2 * S * 3 * 8.0 * S * S
    else:
        n, p, K = case["sequences"], case["order"], case["known"]
        by = 16 * n * (K + case["out"])
        # normal equations, two factorisations, twenty root iterations, the prediction
        fl = n * (8.0 * p * p * (K - K // 2) / 2 + 8.0 * p ** 3 / 3 + 8.0 * 2 * p ** 3 / 3 +
                  20 * 24.0 * p * p + 14.0 * p * (case["out"] - K))
    return {"bytes": float(by), "flops": float(fl)}


# ------------------------------------------------------------------- exact

def _bonds(Lx, Ly):
    r = [(x + Lx * y, (x + 1) % Lx + Lx * y) for y in range(Ly) for x in range(Lx)]
    if Ly > 1:
        r += [(x + Lx * y, x + Lx * ((y + 1) % Ly)) for y in range(Ly) for x in range(Lx)]
    return r


def _hprime64(p, spins, x, lref):
    """(H' v)(s) / psi_ref(s) of the RBM v with parameters p, 64 bits."""
    N, M = x["N"], x["M"]
    th = _theta64(p, spins, N, M)
    V = torch.exp(_logpsi64(p, spins, N, M, th) - lref)
    # v(s^{ij}) = e^{a-part} prod_m 2 cosh(theta_m -+ D_m), relative to psi_ref
    sg = torch.where(th.real < 0, -1.0, 1.0)
    scale = (th * sg).sum(1)
    C, S = 0.5 * (1 + torch.exp(-2 * sg * th)), 0.5 * sg * (1 - torch.exp(-2 * sg * th))
    sd = spins.double()
    base = scale + M * math.log(2.0) - lref
    base = base + torch.complex(sd @ p[:N].real.contiguous(), sd @ p[:N].imag.contiguous())
    W = p[N + M:].reshape(N, M)
    E = torch.zeros(len(spins), dtype=torch.complex128, device="cuda")
    ed = torch.zeros(len(spins), dtype=torch.float64, device="cuda")
    for i, j in _bonds(x["Lx"], x["Ly"]):
        ed += sd[:, i] * sd[:, j]
        k = (spins[:, i] != spins[:, j]).nonzero().squeeze(1)
        si = sd[k, i]
        D = 2 * (W[i] - W[j])
        f = C[k] * torch.cosh(D) - si[:, None] * (S[k] * torch.sinh(D))
        while f.shape[1] > 1:
            if f.shape[1] % 2:
                f = torch.cat([f[:, :-2], f[:, -2:-1] * f[:, -1:]], 1)
                continue
            h = f.shape[1] // 2
            f = f[:, :h] * f[:, h:]
        E[k] += f[:, 0] * torch.exp(-2 * si * (p[i] - p[j]))
    HV = 0.25 * ed * V + 0.5 * torch.exp(base) * E
    return (HV - x["E0"] * V) / x["a"] - WP * V


def _products(s, T):
    """O v and O^dag w without O, 64 bits."""
    sd = s.double()
    N, M = sd.shape[1], T.shape[1]

    def real_mm(a, z):
        return torch.complex(a @ z.real.contiguous(), a @ z.imag.contiguous())

    def ov(v):
        y = real_mm(sd, v[N + M:].reshape(N, M))
        return real_mm(sd, v[:N]) + (T * (y + v[N:N + M])).sum(1)

    def odag(w):
        y = T.conj() * w[:, None]
        return torch.cat([real_mm(sd.T, w), y.sum(0), real_mm(sd.T, y).reshape(-1)])

    return ov, odag


def _force64(spins, T, R, dgamma):
    B = len(spins)
    _, odag = _products(spins, T)
    obar = odag(torch.ones(B, dtype=torch.complex128, device="cuda")).conj() / B
    mR, mRR = R.mean(), (R.abs() ** 2).mean()
    gam = torch.acos(torch.sqrt(torch.clamp(mR.abs() ** 2 / mRR, max=1.0)))
    c = dgamma * torch.where(gam < 1e-8, torch.ones_like(gam), gam / torch.tan(gam))
    return obar, c * (odag(R) / B / mR - obar.conj())


def _cg64(spins, T, F, obar, shift, tol, maxit):
    ov, odag = _products(spins, T)
    x, r = torch.zeros_like(F), F.clone()
    p, rr = r.clone(), (r.abs() ** 2).sum()
    ff = rr.clone()
    for _ in range(maxit):
        u = ov(p)
        Ap = odag(u - (obar * p).sum()) / len(spins) + shift * p
        al = rr / (p.conj() * Ap).sum().real
        x, r = x + al * p, r - al * Ap
        rn = (r.abs() ** 2).sum()
        if not rn > tol * tol * ff:
            break
        p, rr = r + (rn / rr) * p, rn
    return x


def _direct64(spins, T, F, obar, shift):
    """(S + shift) x = F with S from sigma_i sigma_i' (real) times conj(T_j) T_j', in blocks of i."""
    B, N = spins.shape
    M = T.shape[1]
    P = len(F)
    sd = torch.cat([torch.ones(B, 1, dtype=torch.float64, device="cuda"), spins.double()], 1)
    Te = torch.cat([torch.ones(B, 1, dtype=torch.complex128, device="cuda"), T], 1)
    # entry ((i, j), (i', j')) of the extended O = [1, sigma] x [1, T]
    pos = torch.zeros(N + 1, M + 1, dtype=torch.long, device="cuda")
    pos[1:, 0] = torch.arange(N, device="cuda")
    pos[0, 1:] = N + torch.arange(M, device="cuda")
    pos[1:, 1:] = N + M + torch.arange(N * M, device="cuda").reshape(N, M)
    S = torch.empty(P, P, dtype=torch.complex128, device="cuda")
    iu, ju = torch.triu_indices(N + 1, N + 1, device="cuda")
    pair = torch.empty(N + 1, N + 1, dtype=torch.long, device="cuda")
    pair[iu, ju] = pair[ju, iu] = torch.arange(len(iu), device="cuda")
    A = (sd[:, iu] * sd[:, ju]).T.contiguous()
    for j in range(M + 1):
        y = Te[:, j:j + 1].conj() * Te
        G = torch.complex(A @ y.real.contiguous(), A @ y.imag.contiguous()) / B  # [pairs, M + 1]
        i0 = 0 if j else 1
        rows = pos[i0:, j]
        full = G[pair[i0:]]                      # [i, i', j']
        cols = pos.reshape(-1)[1:]               # without the constant (0, 0)
        S[rows[:, None], cols[None, :]] = full.reshape(len(rows), -1)[:, 1:]
    S -= obar.conj()[:, None] * obar[None, :]
    S.diagonal().add_(shift)
    return torch.linalg.solve(S, F)


def _exact_sym(case, seed):
    x = _inputs(case, seed)
    L, N, B = x["Lx"], x["N"], case["B"]
    s = prepare(case, seed)
    spins, lref = s["spins"], s["lp"].to(torch.complex128)
    idx = np.arange(N)
    ks = np.arange(N)
    ph = torch.from_numpy(np.exp(-2j * np.pi * (np.outer(ks % L, idx % L) + np.outer(ks // L, idx // L)) / L)).cuda()
    Bt = torch.empty(N, case["states"], B, dtype=torch.complex128, device="cuda")
    HBt = torch.empty_like(Bt)
    for n in range(case["states"]):
        p = s["params"][n].to(torch.complex128)
        A = torch.zeros(N, B, dtype=torch.complex128, device="cuda")
        HA = torch.zeros_like(A)
        for r in range(4):
            X, Y = idx % L, idx // L
            for _ in range(r):
                X, Y = (L - Y) % L, X
            src = np.stack([(X + m % L) % L + L * ((Y + m // L) % L) for m in range(N)])
            t = spins[:, torch.from_numpy(src).cuda()]          # [B, m, x]
            t = t.permute(1, 0, 2).reshape(N * B, N).contiguous()
            lr = lref.repeat(N)
            A += 0.25 * torch.exp(_logpsi64(p, t, N, x["M"]) - lr).reshape(N, B)
            HA += 0.25 * _hprime64(p, t, x, lr).reshape(N, B)
        Bt[:, n], HBt[:, n] = ph @ A / L, ph @ HA / L
    return [Bt, HBt]


def _exact_krylov(case, seed):
    Bm, HBm = (v.to(torch.complex128) for v in _columns(case, seed))
    B, Nm = case["B"], case["states"]
    G = (Bm.conj() @ Bm.T / B).cpu().numpy()
    H = (Bm.conj() @ HBm.T / B).cpu().numpy()
    H = 0.5 * (H + H.conj().T)
    lam, U = np.linalg.eigh(G)
    keep = lam > 1e-10 * lam.max()
    Gp = (U[:, keep] / lam[keep]) @ U[:, keep].conj().T
    cs = [np.eye(Nm)[0].astype(complex)]
    cs.append(Gp @ (H @ cs[0]))
    for _ in range(2, 2 * Nm):
        cs.append(Gp @ (2.0 * (H @ cs[-1]) - G @ cs[-2]))
    X = U[:, keep] / np.sqrt(lam[keep])
    Hx = X.conj().T @ H @ X
    e, V = np.linalg.eigh(0.5 * (Hx + Hx.conj().T))
    w = np.abs(V.conj().T @ (X.conj().T @ G[:, 0])) ** 2
    pad = np.zeros(Nm - len(e))
    return {"G": G, "H": H, "mu": np.array([(G @ c)[0] for c in cs]), "poles": np.concatenate([e, pad]),
            "weights": np.concatenate([w, pad]), "rank": None}


def _exact_extrapolate(case, seed):
    p, n0, N, n_out = case["order"], case["known"] // 2, case["known"], case["out"]
    out = []
    for mu in _moments(case, seed).cpu().numpy():
        past = np.stack([mu[n - p:n][::-1] for n in range(n0, N)])
        Rm = past.conj().T @ past
        Rm += REG * np.max(np.real(np.diag(Rm))) * np.eye(p)
        a = np.linalg.solve(Rm, -(past.conj().T @ mu[n0:]))
        z = np.roots(np.concatenate([[1.0], a]))
        c = np.linalg.solve(np.vander(z, p, increasing=True).T, mu[N - p:])
        w = np.where(np.abs(z) > 1, z / np.abs(z), z)
        m = np.arange(p, p + n_out - N)
        out.append(np.concatenate([mu, (c[:, None] * w[:, None] ** m).sum(0)]))
    return np.array(out)


def exact(case, seed):
    """The outputs in 64 bits, where the inputs determine them: an iteration, a scan and a sweep
    hang on chains of accept decisions taken in the context's precision and have none."""
    kind = case["kind"]
    if kind in ("iteration", "scan", "sweep"):
        return None
    if kind == "krylov":
        return _exact_krylov(case, seed)
    if kind == "extrapolate":
        return _exact_extrapolate(case, seed)
    if kind == "sym":
        return _exact_sym(case, seed)
    s = prepare(case, seed)
    x = _inputs(case, seed)
    N, M = x["N"], x["M"]
    if kind == "target":
        lref, b = s["lp"].to(torch.complex128), x["beta"]
        E = _hprime64(x["prev"], x["spins"], x, lref)
        return 2 * b[1] * E - b[0] * torch.exp(_logpsi64(x["prev2"], x["spins"], N, M) - lref)
    R = s["R"].to(torch.complex128)
    if kind == "grad":
        th = _theta64(x["cur"], x["spins"], N, M)
        lp = _logpsi64(x["cur"], x["spins"], N, M, th)
        d = lp - s["lp0"].to(torch.complex128)
        w, Ra = torch.exp(2 * d.real), R * torch.exp(-d)
        t, mm = (w * Ra).sum(), (w * Ra.abs() ** 2).sum()
        loss = -torch.log(t.abs() ** 2 / (mm * w.sum()))
        # dL/d conj(log psi_s): the term of |sum w R|^2, of sum w |R|^2 (w |Ra|^2 does not move) and of sum w
        g = 2.0 * (w / w.sum() - w * Ra / t)  # torch's gradient of a real loss is twice that
        _, odag = _products(x["spins"], torch.tanh(th))
        return {"loss": loss, "grad": odag(g)}
    T = s["tanh"].to(torch.complex128)
    obar, F = _force64(x["spins"], T, R, 0.5)
    if case["solver"] == "cg":
        d = _cg64(x["spins"], T, F, obar, case["shift"], 1e-4, 50)
    else:
        d = _direct64(x["spins"], T, F, obar, case["shift"])
    return x["cur"] + d
