"""The workloads that the package's speed is measured on.

Each case is one call (or one whole estimate) through the public entry points with
the sizes of the presets in `paper_2606_09291_gb300.inputs`, the serving mix, the tests
and the benchmark: level gradients in both precisions from the smallest grid to the
largest, plain and allocation-free solves, field synthesis on its own, the
multi-record merge with the optimisation step, and one whole multilevel estimate on
concurrent streams.  `listed()` holds the fixed cases, `draw(rng)` more of the same
ranges; `exact()` evaluates the same quantities in 64 bits with plain torch and numpy
(Philox draws, Karhunen-Loeve field, Jacobi-preconditioned CG, statistics).
"""
import math
import random

import numpy as np
import torch

from paper_2606_09291_gb300 import inputs, mlsgd, serving

# sizes of the workloads: see inputs.PRESETS
_FIELDS = {
    "c1": dict(n_levels=3, n0=8, n_modes=64, corr_len=0.3, sigma=1.0, theta=1.0),
    "c2": dict(n_levels=5, n0=8, n_modes=128, corr_len=0.2, sigma=1.0, theta=10.0),
    "c3": dict(n_levels=4, n0=8, n_modes=256, corr_len=0.2, sigma=1.0, theta=10.0),
    "c4": dict(n_levels=6, n0=8, n_modes=128, corr_len=0.2, sigma=1.0, theta=10.0),
    "c5": dict(n_levels=6, n0=8, n_modes=512, corr_len=0.1, sigma=1.5, theta=100.0),
    "paper": dict(n_levels=4, n0=16, ctrl_level=2, n_modes=125, corr_len=0.15, sigma=1.0, theta=8.0, field_model=1,
                  target_freq=2),
}
_ALPHA = 1e-4


def listed():
    return [
        # a control loop that may not allocate: a few samples of the coarsest grid, FP64
        dict(name="noalloc_fp64_8", kind="solve", preset="c1", precision="fp64", rtol=1e-12, grid=0, samples=4, noalloc=True),
        # level 0 of the plain FP64 gradient at fixed control (64 samples of 8^3)
        dict(name="grad_fp64_l0", kind="grad", preset="c1", precision="fp64", rtol=1e-12, level=0, samples=64),
        # level 1 of the FP64 optimisation run's first batch (16 samples of 16^3 with their 8^3 partners)
        dict(name="grad_fp64_l1", kind="grad", preset="c2", precision="fp64", rtol=1e-10, level=1, samples=16),
        # level 3 of the same run (64^3 with 32^3 partners), an odd adaptive count
        dict(name="grad_fp64_l3", kind="grad", preset="c2", precision="fp64", rtol=1e-10, level=3, samples=9),
        # serving: the coarsest level's request of an estimate (1024 samples of 8^3, control on 256^3)
        dict(name="grad_mixed_l0", kind="grad", preset="c4", precision="mixed", rtol=1e-8, level=0, samples=1024, ir_steps=3),
        # serving: a middle level's request (64 samples of 32^3 with 16^3 partners)
        dict(name="grad_mixed_l2", kind="grad", preset="c4", precision="mixed", rtol=1e-8, level=2, samples=64, ir_steps=3),
        # the batched mixed-precision throughput workload (64^3 with 32^3 partners, 256 modes)
        dict(name="grad_mixed_l3_batch", kind="grad", preset="c3", precision="mixed", rtol=1e-8, level=3, samples=512, ir_steps=0),
        # the top level of the serving mix and of the theta = 100 run: one sample of 256^3
        dict(name="grad_mixed_l5", kind="grad", preset="c4", precision="mixed", rtol=1e-8, level=5, samples=1, ir_steps=3),
        # a state and adjoint solve on the paper's field (64^3), an odd count, FP64 results out
        dict(name="solve_mixed_64", kind="solve", preset="paper", precision="mixed", rtol=1e-8, grid=2, samples=7, noalloc=False),
        # log a of a batch in FP64 (64^3 cells, 256 modes)
        dict(name="field_fp64", kind="field", preset="c3", precision="fp64", level=3, grid=3, samples=64, tc=False),
        # two ranks' records merged on every level, then the step on a 256^3 control
        dict(name="merge_step", kind="step", preset="c4", adaptive=False),
        # one whole multilevel estimate of the serving mix, levels on concurrent streams
        dict(name="serve_mix", kind="serve", preset="c4", mix="1024,256,64,16,4,1"),
    ]


def draw(rng):
    """One more case: samples log-uniform in a range that keeps its work below the largest listed case."""
    kind = rng.choices(["grad64", "gradmx", "solve", "noalloc", "field", "step"], [3, 4, 2, 1, 1.5, 0.5])[0]

    def count(lo, hi):
        return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))

    if kind == "grad64":
        preset = rng.choice(["c1", "c2", "c2", "paper"])
        n0, L = _FIELDS[preset]["n0"], _FIELDS[preset]["n_levels"]
        level = rng.randrange(L)
        N = n0 << level
        return dict(kind="grad", preset=preset, precision="fp64", rtol=rng.choice([1e-10, 1e-12]), level=level,
                    samples=count(1, {8: 300, 16: 130, 32: 40, 64: 8, 128: 1}[N]))
    if kind == "gradmx":
        preset = rng.choice(["c3", "c4", "c5", "paper"])
        n0, L = _FIELDS[preset]["n0"], _FIELDS[preset]["n_levels"]
        level = rng.randrange(L)
        N = n0 << level
        return dict(kind="grad", preset=preset, precision="mixed", rtol=1e-8, level=level,
                    samples=count(1, {8: 2048, 16: 1024, 32: 300, 64: 60, 128: 8, 256: 1}[N]), ir_steps=rng.choice([0, 3]))
    if kind in ("solve", "noalloc"):
        preset = rng.choice(["c1", "c3", "paper"])
        precision = rng.choice(["fp64", "mixed"])
        N0 = _FIELDS[preset]["n0"]
        grid = rng.randrange(2 if kind == "noalloc" else min(_FIELDS[preset]["n_levels"], 4 if N0 == 8 else 3))
        N = N0 << grid
        most = {8: 60, 16: 12, 32: 2}[N] if kind == "noalloc" else {8: 200, 16: 100, 32: 40, 64: 8}[N]
        return dict(kind="solve", preset=preset, precision=precision, rtol=1e-12 if precision == "fp64" else 1e-8, grid=grid,
                    samples=count(1, most), noalloc=kind == "noalloc")
    if kind == "field":
        tc = rng.random() < 0.5
        preset = rng.choice(["c3", "c5"] if tc else ["c1", "c2", "c3", "paper"])
        level = rng.randrange(1, 4 if preset in ("c3", "c5", "c2") else 3)
        N = _FIELDS[preset]["n0"] << level
        return dict(kind="field", preset=preset, precision="mixed" if tc else "fp64", level=level,
                    grid=level - rng.randrange(2), samples=count(1, max(2, min(600, 100 * 64 ** 3 // N ** 3))), tc=tc)
    return dict(kind="step", preset=rng.choice(["c1", "c2", "c3", "paper"]), adaptive=rng.random() < 0.5)


# ---------------------------------------------------------------- inputs
def _config(case):
    c = dict(_FIELDS[case["preset"]], alpha=_ALPHA)
    if "precision" in case:
        c.update(precision=case["precision"], rtol=case.get("rtol", 1e-8), max_iter=50 if case["precision"] == "mixed" else 400)
    if case["kind"] == "grad":
        c.update(max_batch=max(256, case["samples"]), ir_steps=case.get("ir_steps", 0),
                 field_tc=1 if case["precision"] == "mixed" else 0)
    return c


def _ctrl(c):
    return c["n0"] << c.get("ctrl_level", c["n_levels"] - 1)


def _control(Nc, seed, freq=1):
    """A control as the iteration meets it: near the right-hand side of the target, with smooth deviations of a few low
    frequencies (gradients are adjoint averages) and a little sampling noise."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    x = (torch.arange(Nc, dtype=torch.float64, device="cuda") + 0.5) / Nc
    S = torch.stack([torch.sin(m * math.pi * x) for m in range(1, 5)])
    w = torch.randn(4, 4, 4, generator=g, dtype=torch.float64, device="cuda") * 0.1
    w[freq - 1, freq - 1, freq - 1] += 1.0
    z = torch.einsum("abc,az,by,cx->zyx", w, S, S, S) * (3 * (freq * math.pi) ** 2)
    z += 0.02 * torch.randn(Nc, Nc, Nc, generator=g, dtype=torch.float64, device="cuda")
    return z.reshape(-1).contiguous()


def _log_a(case, c, seed):
    """The coefficient a caller of the solve holds: log a of the case's samples, drawn by the library."""
    N = c["n0"] << case["grid"]
    ctx = mlsgd.Context(**dict(c, seed=int(seed)))
    la = torch.empty(case["samples"], N ** 3, dtype=torch.float64, device="cuda")
    ctx.mlsgd_sample_field(int(seed) % 50, case["grid"], case["grid"], 0, case["samples"], log_a=la)
    torch.cuda.synchronize()
    ctx.close()
    return la


def _records(c, seed):
    """Two ranks' level records as a run's first batches leave them: smooth fields that shrink with the level."""
    L, Nc = c["n_levels"], _ctrl(c)
    r = random.Random(int(seed))
    out = []
    for rank in range(2):
        recs = []
        for l in range(L):
            s = 4.0 ** -l
            f = _control(Nc, 977 * int(seed) + 31 * l + rank) * (2e-4 * s)
            phi = 0.06 + 0.01 * r.random()
            sc = [float(8 + r.randrange(1000)), phi, (0.7 if l == 0 else 0.01 * s) * (1 + 0.1 * r.random()),
                  0.3 * s * s * (1 + r.random()), 1e-5 * s * s * (1 + r.random()), phi, 240.0 + r.randrange(1000), 0.0]
            recs.append((f, torch.tensor(sc, dtype=torch.float64, device="cuda")))
        out.append(recs)
    return out


def prepare(case, seed):
    c = _config(case)
    kind = case["kind"]
    if kind == "serve":
        mix = tuple(int(v) for v in case["mix"].split(","))
        cfg, _ = serving.mix_config(case["preset"])
        srv = serving.MixServer(dict(cfg, seed=int(seed)), mix)
        return dict(case=case, srv=srv, z=_control(_ctrl(cfg), seed), request=int(seed) % 50)
    ctx = mlsgd.Context(**dict(c, seed=int(seed)))
    s = dict(case=case, ctx=ctx, it=int(seed) % 50)
    f64 = dict(dtype=torch.float64, device="cuda")
    if kind == "grad":
        s.update(z=_control(_ctrl(c), seed, c.get("target_freq", 1)), stats=ctx.new_stats(case["level"]))
    elif kind == "solve":
        S, nodes = case["samples"], ((c["n0"] << case["grid"]) + 1) ** 3
        s.update(z=_control(_ctrl(c), seed, c.get("target_freq", 1)), la=_log_a(case, c, seed), y=torch.zeros(S, nodes, **f64),
                 q=torch.zeros(S, nodes, **f64), phi=torch.zeros(S, **f64),
                 iters=torch.zeros(S, dtype=torch.int32, device="cuda"), status=torch.zeros(S, dtype=torch.int32, device="cuda"))
    elif kind == "field":
        S, cells = case["samples"], (c["n0"] << case["grid"]) ** 3
        if case["tc"]:
            s.update(la=torch.zeros(S, cells, dtype=torch.float32, device="cuda"),
                     a=torch.zeros(S, cells, dtype=torch.bfloat16, device="cuda"))
        else:
            s.update(xi=torch.zeros(S, c["n_modes"], **f64), la=torch.zeros(S, cells, **f64))
    else:
        Nc = _ctrl(c)
        src = []
        for recs in _records(c, seed):
            rank = []
            for l, (f, sc) in enumerate(recs):
                st = mlsgd.Stats(l, Nc ** 3)
                st.field.copy_(f)
                st.scalars.copy_(sc)
                rank.append(st)
            src.append(rank)
        s.update(src=src, dst=[ctx.new_stats(l) for l in range(c["n_levels"])], z=_control(Nc, seed), grad=torch.zeros(Nc ** 3, **f64),
                 prev=_control(Nc, int(seed) + 5) * 2e-4, tau=0.5 / (_ALPHA + (3 * math.pi ** 2) ** -2))
    return s


# ---------------------------------------------------------------- one pass
def _out(stats):
    """A level record: the mean field; (mean dY, S2 dY, S2 dX); (shift, max Phi); (count, iterations, failures)."""
    s = stats.scalars
    return dict(field=stats.field, mean_dy=s[2], s2_dy=s[3], s2_dx=s[4], phi=torch.stack((s[1], s[5])),
                counts=torch.stack((s[0], s[6], s[7])).to(torch.int64))


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "serve":
        srv = state["srv"]
        srv.submit(state["request"], state["z"])
        return [_out(st) for st in srv.stats]
    ctx = state["ctx"]
    if kind == "grad":
        st = state["stats"]
        ctx.mlsgd_stats_reset(st)
        ctx.mlsgd_level_gradient(state["it"], case["level"], 0, case["samples"], state["z"], st)
        return _out(st)
    if kind == "solve":
        f = ctx.mlsgd_solve_state_adjoint_noalloc if case["noalloc"] else ctx.mlsgd_solve_state_adjoint
        code = f(case["grid"], case["samples"], state["la"], state["z"], state["y"], state["q"], state["phi"], state["iters"],
                 state["status"])
        return dict(y=state["y"], q=state["q"], phi=state["phi"], iters=state["iters"], status=state["status"], code=code)
    if kind == "field":
        if case["tc"]:
            ctx.mlsgd_sample_field_tc(state["it"], case["level"], case["grid"], 0, case["samples"], log_a_f32=state["la"],
                                      a_bf16=state["a"])
            return dict(log_a=state["la"], a=state["a"])
        ctx.mlsgd_sample_field(state["it"], case["level"], case["grid"], 0, case["samples"], xi=state["xi"], log_a=state["la"])
        return dict(xi=state["xi"], log_a=state["la"])
    for l, d in enumerate(state["dst"]):
        ctx.mlsgd_stats_reset(d)
        for rank in state["src"]:
            ctx.mlsgd_stats_merge(d, rank[l])
    if case["adaptive"]:
        rep = ctx.mlsgd_step_adaptive(state["dst"], 1.0, state["tau"], state["z"], state["prev"])
        grad = state["prev"]
    else:
        rep = ctx.mlsgd_step(state["dst"], state["tau"], state["z"], grad=state["grad"])
        grad = state["grad"]
    report = {k: rep[k] for k in ("grad_norm", "risk", "err_sam", "err_num", "tau", "objective", "z_norm")}
    return dict(z=state["z"], grad=grad, report=report, plan=np.array(rep["next_counts"], dtype=np.int64),
                fields=[d.field for d in state["dst"]], scalars=[d.scalars[:5] for d in state["dst"]])


# ---------------------------------------------------------------- the least a pass has to move and compute
# A preconditioned CG iteration cannot do without: reading and writing x, r, p once, reading the coefficient once, and three
# applications of the 21-point operator (the step's and the two smoothing residuals of the V-cycle, whose coarse levels add
# 1/7).  About 12 iterations reach 1e-8, 14 reach 1e-10, 17 reach 1e-12 (per solve), state and adjoint.
def _solve_work(N, S, precision, rtol):
    nodes, cells = (N + 1) ** 3, N ** 3
    el = 4 if precision == "mixed" else 8
    its = 12 if rtol > 1e-9 else (14 if rtol > 1e-11 else 17)
    per = S * (6 * nodes * el + cells * el) * 8 / 7
    flops = S * nodes * (3 * 41 + 20) * 8 / 7
    return 2 * its * per, 2 * its * flops


def _field_work(N, S, K, el):
    return S * (K * 8 + N ** 3 * el), 2.0 * S * (N ** 3 * K ** (1 / 3) * 2 + N * N * K)


def _grad_work(c, precision, rtol, level, S):
    N, Nc = c["n0"] << level, _ctrl(c)
    b, f = 3.0 * Nc ** 3 * 8, 4.0 * Nc ** 3
    for n in (N, N // 2) if level > 0 else (N,):
        for w in (_solve_work(n, S, precision, rtol), _field_work(n, S, c["n_modes"], 4 if precision == "mixed" else 8)):
            b, f = b + w[0], f + w[1]
    return b, f


def work(case):
    c = _config(case)
    kind = case["kind"]
    if kind == "grad":
        b, f = _grad_work(c, case["precision"], case["rtol"], case["level"], case["samples"])
    elif kind == "serve":
        b = f = 0.0
        for l, m in enumerate(int(v) for v in case["mix"].split(",")):
            w = _grad_work(c, "mixed", 1e-8, l, m)
            b, f = b + w[0], f + w[1]
    elif kind == "solve":
        N, S = c["n0"] << case["grid"], case["samples"]
        b, f = _solve_work(N, S, case["precision"], case["rtol"])
        b += S * (N ** 3 * 8 + 2 * (N + 1) ** 3 * 8) + _ctrl(c) ** 3 * 8
    elif kind == "field":
        N, S, K = c["n0"] << case["grid"], case["samples"], c["n_modes"]
        if case["tc"]:
            b, f = S * N ** 3 * 6 + S * K * 2 + N ** 3 * K * 2, 2.0 * S * N ** 3 * K
        else:
            b, f = _field_work(N, S, K, 8)
            b += S * K * 8
    else:
        n, L = _ctrl(c) ** 3, c["n_levels"]
        b, f = 8.0 * n * (L * 3 + 3), n * (L * 8.0 + 8)  # two records in, one out per level; z in and out, the gradient out
    return dict(bytes=float(b), flops=float(f))


# ---------------------------------------------------------------- the same in 64 bits, without the library
def _modes(c):
    """(idx [K, 3], scale [K] = sigma sqrt(lambda), phi(n, x)) of the field."""
    if c.get("field_model", 0) == 1:
        m = round(c["n_modes"] ** (1 / 3))
        # modes (j, k, l), l fastest: cos(j pi x2) cos(k pi x3) cos(l pi x1)
        t = [(l - 1, j - 1, k - 1, math.exp(-math.pi * (j + k + l) * c["corr_len"]))
             for j in range(1, m + 1) for k in range(1, m + 1) for l in range(1, m + 1)]
        return np.array([v[:3] for v in t]), c["sigma"] * np.sqrt([v[3] for v in t]), lambda n, x: np.cos((n + 1) * np.pi * x)
    ci, n1 = 1.0 / c["corr_len"], 64
    om = []
    for m in range(n1):
        lo, hi = m * np.pi / 2, (m + 1) * np.pi / 2
        f = (lambda s: 2 * s * np.sin(s) - ci * np.cos(s)) if m % 2 == 0 else (lambda s: ci * np.sin(s) + 2 * s * np.cos(s))
        flo = f(lo)
        for _ in range(200):
            mid = 0.5 * (lo + hi)
            if mid <= lo or mid >= hi:
                break
            if (f(mid) < 0) == (flo < 0):
                lo = mid
            else:
                hi = mid
        om.append(lo + hi)
    om = np.array(om)
    lam = 2 * ci / (om ** 2 + ci ** 2)
    I = np.stack(np.meshgrid(*[np.arange(n1)] * 3, indexing="ij"), -1).reshape(-1, 3)
    v = np.sort(lam[I], 1)
    key = (v[:, 0] * v[:, 1]) * v[:, 2]
    order = np.lexsort((I[:, 2], I[:, 1], I[:, 0], -key))[:c["n_modes"]]

    def phi(n, x):
        w, t = om[n], x - 0.5
        s = np.sin(w) / (2 * w)
        return np.cos(w * t) / np.sqrt(0.5 + s) if n % 2 == 0 else np.sin(w * t) / np.sqrt(0.5 - s)

    return I[order], c["sigma"] * np.sqrt(key[order]), phi


def _draws(c, seed, it, level, S):
    """xi [S, K]: Philox4x32-10, key = seed, counter = (mode pair, sample, level, iteration)."""
    K = c["n_modes"]
    P = (K + 1) // 2
    M = np.uint64(0xFFFFFFFF)
    ctr = [np.tile(np.arange(P, dtype=np.uint64), S), np.repeat(np.arange(S, dtype=np.uint64), P),
           np.full(S * P, level, np.uint64), np.full(S * P, it, np.uint64)]
    k0, k1 = int(seed) & 0xFFFFFFFF, int(seed) >> 32
    for _ in range(10):
        a, b = ctr[0] * np.uint64(0xD2511F53), ctr[2] * np.uint64(0xCD9E8D57)
        ctr = [(b >> np.uint64(32)) ^ ctr[1] ^ np.uint64(k0), b & M, (a >> np.uint64(32)) ^ ctr[3] ^ np.uint64(k1), a & M]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF

    def uni(h, l):
        return (((h >> np.uint64(5)) << np.uint64(26) | (l >> np.uint64(6))) + np.uint64(1)).astype(np.float64) * 2.0 ** -53

    u1, u2 = uni(ctr[0], ctr[1]), uni(ctr[2], ctr[3])
    if c.get("field_model", 0) == 1:
        v = (-4 + 8 * u1, -4 + 8 * u2)
    else:
        r = np.sqrt(-2 * np.log(u1))
        v = (r * np.cos(2 * np.pi * u2), r * np.sin(2 * np.pi * u2))
    return np.stack(v, -1).reshape(S, 2 * P)[:, :K]


def _field(c, xi, N):
    """log a [S, N, N, N] (z, y, x) at the cell centres."""
    idx, scale, phi = _modes(c)
    x = (np.arange(N) + 0.5) / N
    T = torch.tensor(np.stack([phi(n, x) for n in range(idx.max() + 1)]), device="cuda")
    X, Y, Z = (T[torch.as_tensor(idx[:, d].copy(), device="cuda")] for d in range(3))
    cs = torch.as_tensor(xi * scale, device="cuda")
    yz = (Z[:, :, None] * Y[:, None, :]).reshape(len(scale), -1)
    out = torch.empty(xi.shape[0], N, N, N, dtype=torch.float64, device="cuda")
    for s in range(xi.shape[0]):
        out[s] = ((cs[s][:, None] * yz).t() @ X).reshape(N, N, N)
    return out


def _apply_setup(a):
    """12 (pair sums over a face's two cells) and D = the sum of the eight cells, for interior nodes."""
    N = a.shape[1]
    fxy, fxz, fyz = a[:, :-1] + a[:, 1:], a[:, :, :-1] + a[:, :, 1:], a[:, :, :, :-1] + a[:, :, :, 1:]
    v = fxy[:, :, :-1] + fxy[:, :, 1:]
    return a, fxy, fxz, fyz, 4 * (v[..., :-1] + v[..., 1:]), 1.0 / (12 * N)


def _apply(A, x, out):
    a, fxy, fxz, fyz, D, h = A
    n = a.shape[1]

    def X(w, v, u):
        return x[:, 1 + w:n + w, 1 + v:n + v, 1 + u:n + u]

    o = out[:, 1:-1, 1:-1, 1:-1]
    torch.mul(D, X(0, 0, 0), out=o)
    for p in (0, 1):
        for q in (0, 1):
            u, v = 2 * p - 1, 2 * q - 1
            o.addcmul_(fxy[:, :, q:n - 1 + q, p:n - 1 + p], X(0, v, u), value=-1)
            o.addcmul_(fxz[:, q:n - 1 + q, :, p:n - 1 + p], X(v, 0, u), value=-1)
            o.addcmul_(fyz[:, q:n - 1 + q, p:n - 1 + p, :], X(v, u, 0), value=-1)
            for r in (0, 1):
                o.addcmul_(a[:, r:n - 1 + r, q:n - 1 + q, p:n - 1 + p], X(2 * r - 1, v, u), value=-1)
    o.mul_(h)


def _cg(A, b, rtol=1e-12):
    """Jacobi-preconditioned CG, all samples together, until each is at rtol."""
    dinv = torch.zeros_like(b)
    dinv[:, 1:-1, 1:-1, 1:-1] = 1.0 / (A[4] * A[5])
    x, r, q = torch.zeros_like(b), b.clone(), torch.zeros_like(b)
    z = dinv * r
    p = z.clone()

    def dot(u, v):
        return torch.einsum("sn,sn->s", u.reshape(len(u), -1), v.reshape(len(v), -1)).reshape(-1, 1, 1, 1)

    rz, bb = dot(r, z), dot(b, b)
    for it in range(6000):
        _apply(A, p, q)
        al = torch.nan_to_num(rz / dot(p, q), 0.0, 0.0, 0.0)
        x.addcmul_(al, p)
        r.addcmul_(-al, q)
        if it % 20 == 19 and bool((dot(r, r) <= rtol * rtol * bb).all()):
            break
        torch.mul(dinv, r, out=z)
        rn = dot(r, z)
        p.mul_(torch.nan_to_num(rn / rz, 0.0, 0.0, 0.0)).add_(z)
        rz = rn
    return x


def _ctrl_1d(N, Nc):
    """(W [N+1, Nc], P [Nc, N+1]): int z phi_n and the cell average along one axis."""
    W, P = np.zeros((N + 1, Nc)), np.zeros((Nc, N + 1))
    if Nc >= N:
        r = Nc // N
        for m in range(Nc):
            e, t = m // r, (m % r + 0.5) / r
            P[m, e], P[m, e + 1] = 1 - t, t
        W = P.T / Nc
    else:
        r = N // Nc
        for i in range(N):  # cell i along the axis, parent i // r
            W[i, i // r] += 0.5 / N
            W[i + 1, i // r] += 0.5 / N
            P[i // r, i] += 0.5 / r
            P[i // r, i + 1] += 0.5 / r
    return torch.tensor(W, device="cuda"), torch.tensor(P, device="cuda")


def _tensor3(M, v):
    """M along each axis of v [..., z, y, x]."""
    return torch.einsum("ai,bj,ck,sijk->sabc", M, M, M, v)


def _mass_1d(N):
    m = np.zeros((N + 1, N + 1))
    for i in range(N):
        m[i:i + 2, i:i + 2] += np.array([[2.0, 1.0], [1.0, 2.0]]) / (6 * N)
    return torch.tensor(m, device="cuda")


def _solve_exact(c, log_a, z):
    """y, q [S, n, n, n] and Phi [S]; samples in chunks that fit beside each other."""
    S, N = log_a.shape[0], log_a.shape[1]
    Nc = _ctrl(c)
    W, _ = _ctrl_1d(N, Nc)
    b = _tensor3(W, z.reshape(1, Nc, Nc, Nc))
    inner = torch.zeros_like(b)
    inner[:, 1:-1, 1:-1, 1:-1] = 1.0
    b = b * inner
    g1 = torch.sin(c.get("target_freq", 1) * math.pi * torch.arange(N + 1, dtype=torch.float64, device="cuda") / N)
    g1[0] = g1[-1] = 0.0
    g = g1[:, None, None] * g1[None, :, None] * g1[None, None, :]
    M = _mass_1d(N)
    y = torch.empty(S, N + 1, N + 1, N + 1, dtype=torch.float64, device="cuda")
    q, phi = torch.empty_like(y), torch.empty(S, dtype=torch.float64, device="cuda")
    step = max(1, 64_000_000 // (N + 1) ** 3)
    for s in range(0, S, step):
        A = _apply_setup(torch.exp(log_a[s:s + step]))
        n = A[0].shape[0]
        y[s:s + n] = _cg(A, b.expand(n, -1, -1, -1).contiguous())
        e = y[s:s + n] - g
        me = _tensor3(M, e)
        phi[s:s + n] = 0.5 * (e * me).sum((1, 2, 3))
        q[s:s + n] = _cg(A, me * inner)
    return y, q, phi


def _grad_exact(case, seed):
    c = _config(case)
    level, S, Nc = case["level"], case["samples"], _ctrl(c)
    N, theta = c["n0"] << level, c["theta"]
    z = _control(Nc, seed, c.get("target_freq", 1))
    xi = _draws(c, seed, int(seed) % 50, level, S)
    _, q, phi = _solve_exact(c, _field(c, xi, N), z)
    shift, w = phi.max(), None
    if level > 0:
        _, qc, phic = _solve_exact(c, _field(c, xi, N // 2), z)
        shift = torch.maximum(shift, phic.max())
        up = np.zeros((N + 1, N // 2 + 1))  # the coarse function's values at the fine nodes
        for i in range(N + 1):
            up[i, i // 2] += 0.5
            up[i, (i + 1) // 2] += 0.5
        w = torch.exp(theta * (phic - shift))
        qc = _tensor3(torch.tensor(up, device="cuda"), qc)
    wf = torch.exp(theta * (phi - shift))
    x = wf[:, None, None, None] * q
    dy = wf.clone()
    if level > 0:
        x -= w[:, None, None, None] * qc
        dy -= w
    mean = x.mean(0, keepdim=True)
    _, P = _ctrl_1d(N, Nc)
    d = x - mean
    G = P.t() @ P / Nc
    s2 = (d * _tensor3(G, d)).sum()
    return dict(field=_tensor3(P, mean).reshape(-1), mean_dy=dy.mean(), s2_dy=((dy - dy.mean()) ** 2).sum(), s2_dx=s2,
                phi=torch.stack((shift, shift)), counts=None)


def _step_exact(case, seed):
    c = _config(case)
    theta, Nc, L = c["theta"], _ctrl(c), c["n_levels"]
    hc3 = 1.0 / Nc ** 3
    a, b = _records(c, seed)
    recs = []
    for l in range(L):
        (fa, sa), (fb, sb) = a[l], b[l]
        sa, sb = sa.tolist(), sb.tolist()
        sh = max(sa[1], sb[1])
        wa, wb = math.exp(theta * (sa[1] - sh)), math.exp(theta * (sb[1] - sh))
        na, nb = sa[0], sb[0]
        n = na + nb
        d, dy = fa * wa - fb * wb, sa[2] * wa - sb[2] * wb
        f = fb * wb + (na / n) * d
        recs.append((f, [n, sh, sb[2] * wb + (na / n) * dy, sa[3] * wa ** 2 + sb[3] * wb ** 2 + dy * dy * na * nb / n,
                         sa[4] * wa ** 2 + sb[4] * wb ** 2 + hc3 * float(d.square().sum()) * na * nb / n]))
    cs = max(r[1][1] for r in recs)
    fac = [math.exp(theta * (r[1][1] - cs)) for r in recs]
    ey = sum(f * r[1][2] for f, r in zip(fac, recs))
    ex = sum(f * r[0] for f, r in zip(fac, recs))
    z = _control(Nc, seed)
    g = ex / max(math.exp(-theta * cs), ey) + _ALPHA * z
    gn = math.sqrt(hc3 * float(g.square().sum()))
    risk = cs + math.log(ey) / theta
    zn = math.sqrt(hc3 * float(z.square().sum()))
    c_hat = hc3 * float(ex.square().sum()) / ey ** 2
    err_sam = 0.0
    for f, r in recs:
        err_sam += math.exp(2 * theta * r[1]) * (r[4] + c_hat * r[3]) / (r[0] * (r[0] - 1))
    tau = 0.5 / (_ALPHA + (3 * math.pi ** 2) ** -2)
    if case["adaptive"]:
        prev = _control(Nc, int(seed) + 5) * 2e-4
        lh = math.sqrt(float((g - prev).square().sum())) / (tau * math.sqrt(float(prev.square().sum())))
        t = (gn * gn - err_sam) / (lh * gn * gn)
        tau = t if t > 0 else min(tau, 1.0 / lh)
    report = dict(grad_norm=gn, risk=risk, err_sam=err_sam, err_num=None, tau=tau, objective=risk + 0.5 * _ALPHA * zn * zn, z_norm=zn)
    return dict(z=z - tau * g, grad=g, report=report, plan=None, fields=[r[0] for r in recs],
                scalars=[torch.tensor(r[1], dtype=torch.float64) for r in recs])


def exact(case, seed):
    c, kind = _config(case), case["kind"]
    if kind == "grad":
        return _grad_exact(case, seed)
    if kind == "step":
        return _step_exact(case, seed)
    if kind == "serve":  # six levels of which each has its own case
        return None
    if kind == "solve":
        N = c["n0"] << case["grid"]
        xi = _draws(c, seed, int(seed) % 50, case["grid"], case["samples"])
        y, q, phi = _solve_exact(c, _field(c, xi, N), _control(_ctrl(c), seed, c.get("target_freq", 1)))
        return dict(y=y.reshape(len(y), -1), q=q.reshape(len(q), -1), phi=phi, iters=None, status=None, code=None)
    xi = _draws(c, seed, int(seed) % 50, case["level"], case["samples"])
    la = _field(c, xi, c["n0"] << case["grid"]).reshape(case["samples"], -1)
    if case["tc"]:
        return dict(log_a=la, a=torch.exp(la))
    return dict(xi=torch.as_tensor(xi), log_a=la)
