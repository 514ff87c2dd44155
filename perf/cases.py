"""Performance cases of the PEPS-VMC library: whole cooling steps, Metropolis sweeps, batch
evaluations, direct draws and the fermionic calls, over the sizes, precisions and chain counts
its users run, each one call (or a step's calls) through `paper_2409_05285_gb300.binding`.

A case is a dict of plain values:
  op      step | sweep | eval | direct | fsr | fsweep
  L1, L2, D, chi, J2, prec (fp64 | fp32 | tf32), n (chains or configurations)
  p       sampling exponent (2, or 1 with reweighting)
  graphs  captured launch sequences on a stream of the caller's (peps_set_graphs)
  scale   size of the random entries added to the beta = 0 product state
"""
import math

import numpy as np
import torch

from paper_2409_05285_gb300 import binding, workloads

PREC = {"fp64": binding.PEPS_FP64, "fp32": binding.PEPS_FP32, "tf32": binding.PEPS_TF32}


def _case(name, op, L1, L2, D, chi, n, prec, J2=0.0, p=2, graphs=False, scale=0.1):
    c = dict(op=op, L1=L1, L2=L2, D=D, chi=chi, n=n, prec=prec, J2=J2, p=p, graphs=graphs, scale=scale)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the 4x4 float64 workload (2000 samples per SR step), default stream: one cooling step
        _case("step_4x4_fp64", "step", 4, 4, 2, 4, 2000, "fp64", scale=0.3),
        # a small request of a serving worker: a step of a few chains, launches and latency
        _case("step_4x4_few_chains", "step", 4, 4, 2, 4, 64, "tf32", J2=0.3, p=1, graphs=True, scale=0.3),
        # the 8x8 workload at its full 8192 chains: the cooling step of the headline benchmark
        _case("step_8x8_tf32", "step", 8, 8, 4, 16, 8192, "tf32", graphs=True),
        # Metropolis burn-in of a serving request (1024 chains), reweighted sampling
        _case("sweep_8x8_1024", "sweep", 8, 8, 4, 16, 1024, "tf32", p=1, graphs=True),
        # evaluation of a caller's configurations on the device, all outputs with O rows
        _case("eval_8x8_tf32", "eval", 8, 8, 4, 16, 2048, "tf32"),
        # the J1-J2 10x10 workload's contraction sizes (bond 216 truncated to 36)
        _case("eval_10x10_d6_tf32", "eval", 10, 10, 6, 36, 192, "tf32", J2=0.5),
        # small lattice at a bond its boundary MPS holds exactly (serving sizes, D = 4, chi = D^2)
        _case("eval_4x4_d4_tf32", "eval", 4, 4, 4, 16, 512, "tf32", J2=0.3),
        # the parity path at the 8x8 sizes: float64 check of a mixed-precision run
        _case("eval_8x8_fp64", "eval", 8, 8, 4, 16, 128, "fp64"),
        # float32-level results on a ragged lattice, odd bond and odd batch
        _case("eval_7x5_d3_fp32", "eval", 7, 5, 3, 9, 777, "fp32", J2=0.5, scale=0.2),
        # reweighted direct sampling, double layer of bond D^2 = 4 (6x6, chi = 16)
        _case("direct_6x6_tf32", "direct", 6, 6, 2, 16, 8192, "tf32", scale=0.3),
        # the 6x6 Hubbard workload: an SR step (local energies, O rows, CG) of 128 chains
        _case("fermion_sr_6x6_tf32", "fsr", 6, 6, 4, 16, 128, "tf32"),
        # Metropolis sweep of a small Hubbard lattice in float64
        _case("fermion_sweep_4x3_fp64", "fsweep", 4, 3, 2, 4, 256, "fp64"),
    ]


def draw(rng):
    """One more case of the same ranges; the chain count is cut to what the step of the 8x8
    workload costs."""
    while True:
        op = rng.choice(["step", "step", "sweep", "sweep", "eval", "eval", "eval", "direct", "fsr", "fsweep"])
        fermion = op in ("fsr", "fsweep")
        L1 = rng.randint(3, 5 if fermion else 10)
        L2 = rng.randint(3, 5) if fermion else max(3, min(10, L1 + rng.randint(-2, 2)))
        D = 2 if op == "direct" else rng.choice([2, 3, 4] if fermion else [2, 2, 3, 4, 4, 4, 6])
        prec = "tf32" if D == 6 else rng.choice(["tf32", "tf32", "tf32", "fp32", "fp64"])
        chi = rng.choice([D * D, D * D, rng.randint(D + 1, D * D)])
        if op == "direct":
            chi = rng.randint(6, 16)
        lo, hi = (16, 256) if fermion else (32, 8192)
        n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
        J2 = rng.choice([0.0, round(rng.uniform(0.05, 0.6), 3)]) if not fermion and op != "direct" else 0.0
        c = _case(None, op, L1, L2, D, chi, n, prec, J2, rng.choice([1, 2]), rng.random() < 0.5,
                  {2: 0.3, 3: 0.2}.get(D, 0.1))
        while _seconds(c) > 1.0 and c["n"] > 16:
            c["n"] = c["n"] * 3 // 4
        if _seconds(c) <= 1.0 and c["n"] >= 16:
            return c


# ------------------------------------------------------------------- inputs and passes


def _configs(rng, n, N):
    """Chains as sampled at high temperature: s = s' on most sites, a few per cent not."""
    S = (3 * rng.integers(0, 2, (n, N))).astype(np.uint8)
    off = rng.random((n, N)) < 0.05
    S[off] = rng.integers(0, 4, int(off.sum()))
    return S


def prepare(case, seed):
    c, rng = case, np.random.default_rng(seed)
    L1, L2, D, chi, n, N = c["L1"], c["L2"], c["D"], c["chi"], c["n"], c["L1"] * c["L2"]
    st = dict(op=c["op"], p=c["p"], n=n)
    st["stream"] = torch.cuda.Stream() if c["graphs"] else None
    raw = st["stream"].cuda_stream if c["graphs"] else None
    if c["op"] in ("fsr", "fsweep"):
        st["theta"] = binding.famp_init_theta(L1, L2, D, noise=c["scale"], seed=seed)
        st["S"] = workloads.fermion_support_configs(n, N, seed)
        st["famp"] = binding.FermionAmplitudes(L1, L2, D, chi, n, precision=PREC[c["prec"]], stream=raw)
        st["sweeps"] = 0
        return st
    ctx = binding.Context(L1, L2, D, chi, n, J1=1.0, J2=c["J2"], precision=PREC[c["prec"]], seed=seed,
                          stream=raw)
    st["ctx"], st["theta"] = ctx, workloads.random_theta(L1, L2, D, seed, scale=c["scale"], diag_bias=1.0)
    ctx.set_theta(st["theta"])
    if c["graphs"]:
        ctx.set_graphs(True)
    S = _configs(rng, n, N)
    if c["op"] == "eval":
        f64 = dict(dtype=torch.float64, device="cuda")
        st["S"] = torch.from_numpy(S).cuda()
        st["out"] = dict(log_abs=torch.zeros(n, **f64), sign=torch.zeros(n, dtype=torch.int8, device="cuda"),
                         e_sys=torch.zeros(n, **f64), e_anc=torch.zeros(n, **f64),
                         O=torch.zeros((n, ctx.No), device="cuda",
                                       dtype=torch.float64 if c["prec"] == "fp64" else torch.float32))
        torch.cuda.synchronize()
    elif c["op"] == "direct":
        st["u"] = rng.random((n, N))
    else:
        ctx.set_configs(S)
    return st


def run(st):
    op, n = st["op"], st["n"]
    if op == "step":   # parameters from the host, one cooling step, parameters and chains back
        ctx = st["ctx"]
        ctx.set_theta(st["theta"])
        s = ctx.step(n_sweeps=1, p=st["p"], tau=0.02, eps=1e-4, max_cg=100, cg_tol=1e-10)
        return dict(theta=ctx.get_theta(), S=ctx.get_configs(), E=s["E_site"], E_err=s["E_err"],
                    chi=s["chi_sus"], accept=s["accept"], diag=s["diag_frac"], cg=s["cg_iters"])
    if op == "sweep":
        st["ctx"].mc_sweep(1, p=st["p"])
        return st["ctx"].get_configs()
    if op == "eval":
        o = st["out"]
        st["ctx"].eval_batch_device(st["S"], o["log_abs"], o["sign"], o["e_sys"], o["e_anc"], o["O"])
        return o
    if op == "direct":
        logq = st["ctx"].direct_draw(st["u"], b_d=0.98, exponent=0.5)
        return dict(log_q=logq, S=st["ctx"].get_configs())
    if op == "fsr":
        th, s = st["famp"].sr_step(st["theta"], st["S"], 1.0, 8.0, 4.0, p=st["p"], tau=0.02)
        return dict(theta=th, E=s["E_site"], E_err=s["E_err"], docc=s["docc"], density=s["density"],
                    cg=s["cg_iters"])
    S, acc, la, sg = st["famp"].sweep(st["theta"], st["S"], p=st["p"], seed=7, sweep0=st["sweeps"])
    st["S"], st["sweeps"] = S, st["sweeps"] + 1
    return dict(S=S, accepted=acc, log_abs=la, sign=sg)


# ------------------------------------------------------------------- work of one pass


def _bonds(L1, L2, J2):
    b = [(r * L2 + q, r * L2 + q + 1, 1.0) for r in range(L1) for q in range(L2 - 1)]
    b += [(r * L2 + q, r * L2 + q + L2, 1.0) for r in range(L1 - 1) for q in range(L2)]
    if J2:
        for i in (r * L2 + q for r in range(L1 - 1) for q in range(L2 - 1)):
            b += [(i, i + L2 + 1, J2), (i + 1, i + L2, J2)]
    return b


def _flops(L1, L2, D, chi, J2=0.0):
    """(environments, one strip of each row and row pair, evaluation of all ratios and O) flops
    of one configuration: contractions at the bonds the boundary MPS needs, truncations not
    counted."""
    env = strip = ratios = 0.0
    for r in range(L1):
        up = [min(chi, D ** min(r, q, L2 - q)) for q in range(L2 + 1)]
        dn = [min(chi, D ** min(L1 - 1 - r, q, L2 - q)) for q in range(L2 + 1)]
        d2 = [min(chi, D ** min(max(L1 - 2 - r, 0), q, L2 - q)) for q in range(L2 + 1)]
        u, d = (1 if r == 0 else D), (1 if r == L1 - 1 else D)
        d3 = 1 if r + 1 == L1 - 1 else D
        for q in range(L2):
            l, g = (1 if q == 0 else D), (1 if q == L2 - 1 else D)
            a, x, b, y = up[q], up[q + 1], dn[q], dn[q + 1]
            env += 2.0 * (a * x + b * y) * l * g * u * d
            one = 2.0 * (l * b * u * x * a + b * x * g * d * l * u + x * g * y * b * d)
            strip += 2 * one
            ratios += 4 * one + 2.0 * (l * b * u * g * y * x + l * g * u * d * b * y)
            if r + 1 < L1:
                b, y = d2[q], d2[q + 1]
                two = 2.0 * (l * l * b * u * x * a + l * b * x * g * d * l * u + b * x * g * g * d3 * l * d +
                             x * g * g * y * b * d3)
                strip += 2 * two
                ratios += (10 if J2 else 2) * two
    return env, strip, ratios


def work(case):
    c = case
    L1, L2, D, chi, n, op = c["L1"], c["L2"], c["D"], c["chi"], c["n"], c["op"]
    N, w = L1 * L2, 8 if c["prec"] == "fp64" else 4
    No = workloads.n_params(L1, L2, D) // 4
    env, strip, ratios = _flops(L1, L2, D, chi, c["J2"])
    if op == "eval":
        return dict(bytes=n * (N + 25) + 4 * No * 8 + n * No * w, flops=n * (env + strip + ratios))
    if op == "sweep":
        return dict(bytes=2 * n * N + 4 * No * 8, flops=n * (env + strip + ratios))
    if op == "step":
        return dict(bytes=2 * n * N + 2 * 4 * No * 8, flops=n * (2 * (env + strip + ratios) + 4.0 * No * 100))
    if op == "direct":
        env, strip, _ = _flops(L1, L2, D * D, chi)
        return dict(bytes=n * (9 * N + 8) + 4 * No * 8, flops=n * (env + 3 * strip))
    pairs = 2 * N + 4 * (2 * N - L1 - L2)
    if op == "fsweep":   # every proposal one environment pass and one row's strip
        return dict(bytes=2 * n * N + 16 * No * 8, flops=n * pairs / 2 * (env + strip / L1))
    return dict(bytes=n * N + 2 * 16 * No * 8, flops=n * (pairs / 2 * (env + strip / L1) + strip + 4.0 * No * 50))


def _seconds(c):
    """Rough duration of a pass, for choosing the sizes of drawn cases."""
    rate = {"tf32": 3.5e12, "fp32": 1.2e12, "fp64": 6e10}[c["prec"]] / (4.0 if c["D"] in (3, 5) else 1.0)
    N = c["L1"] * c["L2"]
    launches = {"step": 130, "sweep": 70, "eval": 70, "direct": 110, "fsr": 3000, "fsweep": 1300}[c["op"]] * N
    trunc = 2e-9 * N * c["n"] * c["chi"] * c["D"] ** 2 * (8 if c["prec"] == "fp64" else 1)
    return work(c)["flops"] / rate + launches * (2 if c["J2"] else 1) * 8e-6 + trunc


# ------------------------------------------------------------------- values in 64 bits


def _amplitude(A, L1, L2):
    """(log|rho|, sign) of m configurations: A[site] is [m][dl][dr][du][dd]; exact contraction,
    one site at a time into the row of open legs."""
    m = A[0].shape[0]
    v, log = torch.ones((m, 1), dtype=torch.float64, device=A[0].device), 0.0
    for r in range(L1):
        cur, P = v.reshape(m, 1, -1, 1), 1
        for q in range(L2):
            a = A[r * L2 + q]
            l, g, u, d = a.shape[1:]
            t = cur.reshape(m, P, u, -1, l).permute(0, 1, 3, 4, 2).reshape(m, -1, l * u)
            t = torch.bmm(t, a.permute(0, 1, 3, 4, 2).reshape(m, l * u, d * g))
            P *= d
            cur = t.reshape(m, P // d, -1, d, g).permute(0, 1, 3, 2, 4)
        v = cur.reshape(m, P)
        s = v.detach().abs().amax(1, keepdim=True)
        v, log = v / s, log + s[:, 0].log()
    return v[:, 0].abs().log() + log, v[:, 0].sign()


def exact(case, seed):
    """log|rho|, sign, E_sys, E_anc and O of the evaluated configurations by exact contraction,
    where chi holds every bond of the network's boundary (else the result is chi's own)."""
    c = case
    L1, L2, D, N, n = c["L1"], c["L2"], c["D"], c["L1"] * c["L2"], c["n"]
    if c["op"] != "eval" or c["chi"] < D ** min(L1 - 1, L2 // 2) or D ** L2 > 2048:
        return None
    bonds = _bonds(L1, L2, c["J2"])
    if n * len(bonds) * N * D ** (L2 + 3) * 4.0 > 4e12:
        return None
    theta = torch.from_numpy(workloads.random_theta(L1, L2, D, seed, scale=c["scale"], diag_bias=1.0)).cuda()
    if c["prec"] != "fp64":   # the network that the float32 paths hold
        theta = theta.float().double()
    T, off = [], 0
    for d in workloads.site_dims(L1, L2, D):
        sz = 4 * int(np.prod(d))
        T.append(theta[off:off + sz].reshape(4, *d))
        off += sz
    S = torch.from_numpy(_configs(np.random.default_rng(seed), n, N)).cuda().long()
    step = max(1, (1 << 25) // D ** (L2 + 1))

    def amps(X):
        out = [_amplitude([T[i][x[:, i]] for i in range(N)], L1, L2) for x in X.split(step)]
        return torch.cat([o[0] for o in out]), torch.cat([o[1] for o in out])

    la, sg, O = [], [], []
    for x in S.split(max(1, step // 4)):
        A = [T[i][x[:, i]].requires_grad_(True) for i in range(N)]
        l, s = _amplitude(A, L1, L2)
        l.sum().backward()
        la.append(l.detach()), sg.append(s.detach())
        O.append(torch.cat([a.grad.reshape(x.shape[0], -1) for a in A], 1))
    la, sg, O = torch.cat(la), torch.cat(sg), torch.cat(O)
    E = []
    for shift in (1, 0):   # system spins (bit 1), ancilla spins (bit 0)
        s = (S >> shift) & 1
        e = torch.zeros(n, dtype=torch.float64, device="cuda")
        for i, j, J in bonds:
            e += J * (0.5 - s[:, i]) * (0.5 - s[:, j])
            k = torch.nonzero(s[:, i] != s[:, j])[:, 0]
            if k.numel():
                X = S[k].clone()
                X[:, i] ^= 1 << shift
                X[:, j] ^= 1 << shift
                l2, s2 = amps(X)
                e[k] += 0.5 * J * s2 * sg[k] * (l2 - la[k]).exp()
        E.append(e)
    return dict(log_abs=la, sign=sg.to(torch.int8), e_sys=E[0], e_anc=E[1],
                O=O)
