"""What this library is used for, as calls to measure: one dict per case.

A case names a kind of call, a lattice (Lx x Ly sites, M slices of dtau), a
number of chains or configurations B and the options of the call.  The
kinds are the steps of self-learning determinantal Monte Carlo as a program
runs them, through the binding's public calls:

  weight  log|det| and sign of one flavour for B configurations
  green   the equal-time Green's functions of B configurations
  logw    the exact log weight (both flavours and the bare part)
  sweep   one local DQMC sweep of B chains (step i: training data)
  fit     the effective model fitted to n configurations (step ii)
  eff     sweeps of the effective model (step iii)
  step    one cumulative update of B chains (steps iii and iv)
  uneven  one replay of a graph of chains on several lattices
"""
import math

import numpy as np
import torch

from paper_1612_03804_gb300 import effmodel, sldqmc

T_HOP, J_ISING, FIELD = 1.0, 1.0, 2.774
CLASSES = {4: effmodel.CLASSES_4, 16: effmodel.paper_classes()}


def _case(kind, Lx, Ly, M, B, dtau=0.05, n_wrap=10, mu=-0.5, xi=1.0, prec="fp64", **more):
    return dict(kind=kind, Lx=Lx, Ly=Ly, M=M, B=B, dtau=dtau, n_wrap=n_wrap, mu=mu, xi=xi, prec=prec, **more)


def listed():
    c = [
        # one configuration of the smallest lattice: plain FP64 DQMC at beta = 2, latency only
        ("weight_4x4", _case("weight", 4, 4, 20, 1, dtau=0.1, mu=0.0)),
        # training data: local sweeps of 64 chains on 8x8 at beta = 8
        ("sweep_8x8", _case("sweep", 8, 8, 160, 64, rank=1)),
        # local sweeps at the critical temperature (beta = 1), immediate updates
        ("sweep_16x16", _case("sweep", 16, 16, 20, 16, n_wrap=20, rank=1)),
        # the same on a larger lattice, delayed rank-32 updates
        ("sweep_24x24", _case("sweep", 24, 24, 20, 8, n_wrap=20, rank=32)),
        # Green's functions for measurements, N = 400 (not a multiple of 32), mid-chain slice
        ("green_20x20", _case("green", 20, 20, 80, 4, eta=-1, tau=37)),
        # 128 production chains on 16x16 at beta = 8, split TF32, n_wrap as the autotuner picks it
        ("step_16x16", _case("step", 16, 16, 160, 128, n_wrap=32, prec="3xtf32", classes=4, n_eff=1, form="dense")),
        # single-flavour weights on 32x32 at beta = 10, split BF16
        ("weight_32x32", _case("weight", 32, 32, 200, 4, prec="bf16x3", eta=-1)),
        # exact log weight with the separable propagator
        ("logw_separable", _case("logw", 32, 32, 100, 4, dtau=0.1, prec="3xtf32", form="separable")),
        # the largest lattice, a short chain of one configuration
        ("weight_100x100", _case("weight", 100, 100, 20, 1, dtau=0.1, prec="3xtf32", eta=1)),
        # ten sweeps of the 16-coupling model between two exact weights
        ("eff_24x24", _case("eff", 24, 24, 20, 16, classes=16, n_sweeps=10)),
        # the fit of the effective model on 8x8 training configurations, weights included
        ("fit_8x8", _case("fit", 8, 8, 20, 64, n_wrap=20, classes=4, n=512)),
        # chains of several lattices stepped by one graph
        ("uneven", _case("uneven", 12, 12, 80, 4, prec="3xtf32", lattices="12,16,20,24,32", classes=4, n_eff=1)),
    ]
    return [dict(d, name=n) for n, d in c]


def draw(rng):
    """One more case of the same ranges."""
    def size(lo, hi):  # spread over the logarithm
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def lattice(lo, hi):
        Lx = size(lo, hi)
        return Lx, min(hi, max(lo, Lx + rng.choice((-3, -2, -1, 0, 0, 0, 1, 2, 3))))

    def budget(Lx, Ly, M, B, n3, limit=1.5e11):
        # chains and slices scaled down until n3 N^3 operations per slice and chain fit the limit
        per = n3 * float(Lx * Ly) ** 3
        B = max(1, min(B, int(limit / (per * M))))
        return max(2, min(M, int(limit / (per * B)))), B

    kind = rng.choice(("weight", "weight", "green", "logw", "sweep", "sweep", "fit", "eff", "step", "step", "uneven"))
    dtau, mu = rng.choice((0.05, 0.1)), rng.choice((0.0, -0.5, -0.5, 0.3))
    n_wrap = rng.choice((4, 5, 8, 10, 10, 16)) if dtau > 0.08 else rng.choice((5, 8, 10, 16, 20, 32))
    M, kw = size(20, 200), dict(dtau=dtau, mu=mu, n_wrap=n_wrap)
    if kind in ("weight", "logw", "step") and rng.random() < 0.6:
        prec = rng.choice(("3xtf32", "3xtf32", "bf16x3", "bf16"))
        Lx, Ly = lattice(12, 64)
        M, B = budget(Lx, Ly, M, size(1, 128), 2.0, 1.5e13)
    else:
        prec = "fp64"
        Lx, Ly = lattice(4, 24)
        M, B = budget(Lx, Ly, M, size(1, 128), {"sweep": 16.0, "green": 6.0}.get(kind, 4.0))
    kw["prec"] = prec
    if kind == "weight":
        return _case(kind, Lx, Ly, M, B, eta=rng.choice((1, -1)), form=rng.choice(("dense", "dense", "separable")), **kw)
    if kind == "green":
        return _case(kind, Lx, Ly, M, B, eta=rng.choice((1, -1)), tau=rng.randrange(M + 1), **kw)
    if kind == "logw":
        return _case(kind, Lx, Ly, M, B, form=rng.choice(("dense", "separable")), **kw)
    if kind == "sweep":
        rank = rng.choice((1, 8, 32, 32)) if Lx * Ly > 100 else rng.choice((1, 1, 16))
        while True:  # a sweep recomputes G from all M slices every n_wrap slices: shorter chains until about 0.6 s
            c = _case(kind, Lx, Ly, M, B, rank=rank, **kw)
            blocks = math.ceil(M / n_wrap)
            chain = M * 40e-6 + blocks * (1 + Lx * Ly // 32) * 150e-6
            if M <= 10 or 2 * blocks * chain + M * Lx * Ly * 8e-6 + work(c)["flops"] / 8e11 < 0.6:
                return c
            M = int(0.85 * M)
    if kind == "step":
        return _case(kind, Lx, Ly, M, B, classes=rng.choice((4, 16)), n_eff=rng.choice((1, 1, 10)),
                     form=rng.choice(("dense", "dense", "separable")), **kw)
    if kind == "fit":
        Lx, Ly = lattice(4, 8)
        return _case(kind, Lx, Ly, size(20, 40), size(16, 64), classes=rng.choice((4, 16)), n=size(64, 1000), **kw)
    if kind == "eff":
        Lx, Ly = lattice(8, 100)
        M = size(20, 100)
        return _case(kind, Lx, Ly, M, max(1, min(size(1, 128), 4000000 // (Lx * Ly * M))), classes=rng.choice((4, 16)),
                     n_sweeps=size(1, 10), **kw)
    kw["prec"] = "3xtf32"
    some = sorted(rng.sample((12, 13, 16, 18, 20, 22, 24, 28, 32), rng.randint(2, 4)))
    return _case("uneven", some[0], some[0], size(20, 100), size(1, 8), lattices=",".join(map(str, some)), classes=4,
                 n_eff=1, **kw)


def _fields(case, seed, count, L=None):
    """Domain fields of +-1 (int8, count x M x N) as chains near the ordering
    temperature hold them: the sign of Gaussian noise smoothed over three
    sites and a quarter of the slices, with one site in twenty flipped."""
    Lx, Ly = (L, L) if L else (case["Lx"], case["Ly"])
    M = case["M"]
    g = torch.Generator(device="cuda").manual_seed(int(seed) * 1009 + Lx)
    x = torch.randn((count, M, Ly, Lx), generator=g, device="cuda")
    for axis, width in ((1, max(1, M // 4)), (2, min(3, Ly)), (3, min(3, Lx))):
        n = x.shape[axis]
        c = torch.cat([x, x.narrow(axis, 0, width)], dim=axis).cumsum(axis, dtype=torch.float64)
        x = (c.narrow(axis, width, n) - c.narrow(axis, 0, n)).float()
    flip = torch.rand(x.shape, generator=g, device="cuda") < 0.05
    return torch.where((x >= 0) ^ flip, 1, -1).to(torch.int8).reshape(count, M, Lx * Ly).contiguous()


def _couplings(case):
    """The bare Ising action as couplings of the case's classes (nearest
    neighbours in space and in time), with small longer-ranged ones."""
    beta, dtau = case["M"] * case["dtau"], case["dtau"]
    kt = -0.5 * math.log(math.tanh(dtau * FIELD))
    J = np.full(case["classes"], 1e-3 * dtau / beta)
    J[0], J[3 if case["classes"] == 4 else 2] = -dtau * J_ISING / beta, -kt / beta
    return J


def _context(case, L=None):
    c = sldqmc.Context(L or case["Lx"], L or case["Ly"], t=T_HOP, mu=case["mu"], xi=case["xi"],
                       beta=case["M"] * case["dtau"], dtau=case["dtau"], n_wrap=min(case["n_wrap"], case["M"]), J=J_ISING,
                       h=FIELD, prec=case["prec"], max_batch=case["B"])
    if "classes" in case:
        c.set_effective_model(CLASSES[case["classes"]], _couplings(case))
    if case.get("form") == "separable":
        c.set_kinetic_form("separable")
    if case.get("rank", 1) > 1:
        c.set_local_update_rank(case["rank"])
    return c


_streams = []


def _graph_stream():
    """The one stream that a program's graphs are launched on."""
    if not _streams:
        _streams.append(torch.cuda.Stream())
    return _streams[0]


class _State:
    pass


def prepare(case, seed):
    st = _State()
    st.case, st.seed, st.step, kind, B = case, int(seed), 0, case["kind"], case["B"]
    f64 = dict(dtype=torch.float64, device="cuda")
    if kind == "uneven":
        st.members = []
        for k, L in enumerate(int(v) for v in case["lattices"].split(",")):
            ctx, s = _context(case, L), _fields(case, seed, B, L)
            lw, acc = torch.zeros(B, **f64), torch.zeros(B, dtype=torch.int32, device="cuda")
            ctx.log_weight_batch_dev(s, lw)
            ctx.sync()
            st.members.append((ctx, s, lw, acc, 7000 + k + 100 * st.seed))
        st.graph = sldqmc.Graph(st.members, n_eff=case["n_eff"], step0=0, stream=_graph_stream().cuda_stream)
        return st
    st.ctx = _context(case)
    if kind == "fit":
        st.cfgs = _fields(case, seed, case["n"]).cpu().numpy()
        return st
    st.s = _fields(case, seed, B)
    if kind in ("weight", "green", "logw", "step"):
        st.ld, st.sign = torch.zeros(B, **f64), torch.zeros(B, dtype=torch.int32, device="cuda")
    if kind == "green":
        st.G = torch.zeros((B, st.ctx.N, st.ctx.N), **f64)
    if kind == "step":
        st.acc = torch.zeros(B, dtype=torch.int32, device="cuda")
        st.ctx.log_weight_batch_dev(st.s, st.ld)
    if kind == "eff":
        st.acc = torch.zeros(B, dtype=torch.int64, device="cuda")
    return st


def run(st):
    c, kind = st.case, st.case["kind"]
    if kind == "weight":
        st.ctx.weight_batch_dev(st.s, c.get("eta", -1), st.ld, st.sign)
        return st.ld, st.sign
    if kind == "green":
        st.ctx.green_batch_dev(st.s, c["eta"], c["tau"], st.G, st.ld, st.sign)
        return st.G, st.ld, st.sign
    if kind == "logw":
        st.ctx.log_weight_batch_dev(st.s, st.ld)
        return st.ld
    if kind == "fit":
        st.ctx.set_effective_model(CLASSES[c["classes"]], _couplings(c))  # the classes to fit
        J, E0, r2 = st.ctx.fit_effective_action(st.cfgs)
        return J, E0, r2
    if kind == "uneven":
        st.graph.launch(1)
        return [(m[1], m[2], m[3]) for m in st.members]
    st.step += 1
    if kind == "sweep":  # the chains move on from where the last sweep left them
        st.ctx.local_sweep_batch_dev(st.s, 17 + st.seed, st.step, 1, want_stats=False)
        return st.s
    if kind == "eff":
        st.ctx.eff_sweeps_batch_dev(st.s, c["n_sweeps"], 23 + st.seed, st.step, -1, st.acc)
        return st.s, st.acc
    st.ctx.cumulative_batch_dev(st.s, st.ld, c["n_eff"], 29 + st.seed, st.step, 1, st.acc)
    return st.s, st.ld, st.acc


def _weight_flops(case, N):
    """Dense (or separable) slice products, 11/3 N^3 per stabilised block, 2/3 N^3 for the determinant."""
    slice_flops = 2.0 * N * N * ((case["Lx"] + case["Ly"]) if case.get("form") == "separable" else N)
    return case["M"] * slice_flops + (11.0 / 3.0 * math.ceil(case["M"] / case["n_wrap"]) + 2.0 / 3.0) * N ** 3


def work(case):
    kind, B, M, N = case["kind"], case["B"], case["M"], case["Lx"] * case["Ly"]
    field = float(B * M * N)
    n_off = sum(len(c) for c in CLASSES[case.get("classes", 4)])
    eff = field * n_off * 4.0  # two neighbours of each offset, read and added
    if kind == "weight":
        return {"bytes": field + 12.0 * B, "flops": B * _weight_flops(case, N)}
    if kind == "green":
        return {"bytes": field + 8.0 * B * N * N, "flops": B * (_weight_flops(case, N) + 2.0 * N ** 3)}
    if kind == "logw":
        return {"bytes": field + 8.0 * B, "flops": 2.0 * B * _weight_flops(case, N)}
    if kind == "fit":
        return {"bytes": float(case["n"] * M * N), "flops": 2.0 * case["n"] * _weight_flops(case, N)}
    if kind == "eff":
        return {"bytes": 2.0 * field, "flops": case["n_sweeps"] * eff}
    if kind == "step":
        return {"bytes": 2.0 * field, "flops": 2.0 * B * _weight_flops(case, N) + case["n_eff"] * eff}
    if kind == "uneven":
        Ls = [int(v) for v in case["lattices"].split(",")]
        return {"bytes": 2.0 * sum(B * M * L * L for L in Ls), "flops": sum(2.0 * B * _weight_flops(case, L * L) for L in Ls)}
    # sweep: per slice the wrap of both flavours (two products each) and a rank-1
    # update per accepted flip (about one site in ten); a fresh G every n_wrap slices
    fresh = 2.0 * math.ceil(M / case["n_wrap"]) * (_weight_flops(case, N) + 2.0 * N ** 3)
    return {"bytes": 2.0 * field, "flops": B * (M * (8.0 * N ** 3 + 0.4 * N ** 3) + fresh)}


# ------------------------------------------------------------ in 64 bits
def _expm(case, sign):
    """exp(sign dtau K) for K = -t A - mu 1 on the periodic lattice, by eigenvectors."""
    Lx, Ly = case["Lx"], case["Ly"]

    def ring(L):
        A = torch.zeros((L, L), dtype=torch.float64)
        for x in range(L):
            if L > 1:
                A[x, (x + 1) % L] += 1.0
                A[(x + 1) % L, x] += 1.0
        return A

    K = -T_HOP * (torch.kron(torch.eye(Ly, dtype=torch.float64), ring(Lx))
                  + torch.kron(ring(Ly), torch.eye(Lx, dtype=torch.float64)))
    w, v = torch.linalg.eigh(K - case["mu"] * torch.eye(Lx * Ly, dtype=torch.float64))
    return (v * torch.exp(sign * case["dtau"] * w)) @ v.T


def _exact_det(case, s, eta, tau=0, want_G=False):
    """log|det(1 + B_tau .. B_1 B_M .. B_tau+1)|, its sign and the inverse for
    the fields s (B x M x N): the product kept as Q diag(d) T by QR every half
    unit of imaginary time, d split into its large and small parts at the end."""
    dev = "cuda" if torch.cuda.is_available() and s.shape[-1] > 64 else "cpu"
    E = _expm(case, -1.0).to(dev)
    s = s.to(dev, torch.float64)
    n, M, N = s.shape
    Q = torch.eye(N, dtype=torch.float64, device=dev).expand(n, N, N)
    d, T = torch.ones((n, N), dtype=torch.float64, device=dev), Q
    X, every = Q, max(1, round(0.5 / case["dtau"]))
    for k in range(M):
        X = E @ (torch.exp(eta * case["dtau"] * case["xi"] * s[:, (tau + k) % M])[:, :, None] * X)
        if (k + 1) % every == 0 or k == M - 1:
            X = X * d[:, None, :]
            order = torch.argsort(X.norm(dim=1), dim=1, descending=True)
            Q, R = torch.linalg.qr(torch.gather(X, 2, order[:, None, :].expand(-1, N, -1)))
            d = torch.diagonal(R, dim1=1, dim2=2).abs()
            T = (R / d[:, :, None]) @ torch.gather(T, 1, order[:, :, None].expand(-1, -1, N))
            X = Q
    big, small = torch.clamp(d, min=1.0), torch.clamp(d, max=1.0)
    left = Q.transpose(1, 2) / big[:, :, None]
    mid = left + small[:, :, None] * T
    sg, ld = torch.linalg.slogdet(mid)
    sign = (sg * torch.linalg.slogdet(Q)[0]).to(torch.int32)
    return ld + torch.log(big).sum(1), sign, torch.linalg.solve(mid, left) if want_G else None


def _exact_logw(case, s):
    x = s.to(torch.float64).reshape(s.shape[0], case["M"], case["Ly"], case["Lx"])
    dtau = case["dtau"]
    space = sum((x * torch.roll(x, 1, dims=a)).sum((1, 2, 3)) for a, L in ((2, case["Ly"]), (3, case["Lx"])) if L > 1)
    time = (x * torch.roll(x, 1, dims=1)).sum((1, 2, 3))
    bare = dtau * J_ISING * space - 0.5 * math.log(math.tanh(dtau * FIELD)) * time
    return sum(2.0 * _exact_det(case, s, eta)[0].cpu() for eta in (1, -1)) + bare.cpu()


def _exact_fit(case, s):
    x = s.cpu().numpy().astype(np.float64).reshape(s.shape[0], case["M"], case["Ly"], case["Lx"])
    F = np.stack([sum((x * np.roll(x, (-o[2], -o[1], -o[0]), axis=(1, 2, 3))).sum((1, 2, 3)) for o in c)
                  for c in CLASSES[case["classes"]]], axis=1)
    y = _exact_logw(case, s).numpy()
    keep = F.std(axis=0) > 0
    A = np.concatenate([np.ones((len(y), 1)), (F - F.mean(0)) / np.where(keep, F.std(0), 1.0)], axis=1)
    if np.linalg.cond(A) > 1e6:
        return None
    x, beta = np.linalg.lstsq(A, y, rcond=None)[0], case["M"] * case["dtau"]
    a = x[1:] / F.std(0)
    r = y - A @ x
    return -a / beta, float(-(x[0] - a @ F.mean(0)) / beta), float(1.0 - (r @ r) / ((y - y.mean()) ** 2).sum())


def exact(case, seed):
    kind, N = case["kind"], case["Lx"] * case["Ly"]
    if kind not in ("weight", "green", "logw", "fit"):
        return None  # moves of Markov chains: whole numbers decided one after another
    count = case["n"] if kind == "fit" else case["B"]
    flavours = 2 if kind in ("logw", "fit") else 1
    if flavours * count * case["M"] * (2.0 * N ** 3 / 8e11 + N * N / 2e7 * case["dtau"] / 0.5) > 20.0:
        return None  # the products and the factorisations would take over 20 seconds
    s = _fields(case, seed, count)
    if kind == "weight":
        ld, sign, _ = _exact_det(case, s, case.get("eta", -1))
        return ld, sign
    if kind == "green":
        ld, sign, G = _exact_det(case, s, case["eta"], case["tau"] % case["M"], True)
        return G, ld, sign
    return _exact_logw(case, s) if kind == "logw" else _exact_fit(case, s)
