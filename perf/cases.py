"""What the solver is timed on: the calls a user's program makes, over the range of sizes it makes them at.

Twelve listed cases, each one pass through the public entry points of the package.  Inputs are drawn on the spot
from the seed, with the distributions of the workloads in lpgen (dense integer, dense real with 10% zeros,
degenerate, general right-hand sides, batches of small LPs, a family of perturbed instances).
"""
import math

import numpy as np
import torch

from paper_1803_04378_gb300 import lpgb


def listed():
    return [
        # one small dense LP, solved again and again: launches and latencies
        dict(name="lp_int_200x200", what="lp", family="int", m=200, n=200),
        # a mid-size dense LP of odd sizes from its slack basis
        dict(name="lp_real_701x1203", what="lp", family="real", m=701, n=1203),
        # the headline problem: one large dense LP from the slack basis to its optimum
        dict(name="lp_real_4096x8192", what="lp", family="real", m=4096, n=8192),
        # every pivot degenerate: the tabu list and the safety net at work
        dict(name="lp_degenerate_256x512", what="lp", family="degenerate", m=256, n=512),
        # negative right-hand sides: Phase I, then Phase II
        dict(name="lp_general_200x300", what="lp", family="general", m=200, n=300),
        # a new instance of a family in a handle that is there: data in, cold solve, solution out
        dict(name="family_cold_1024x2048", what="family", warm=False, m=1024, n=2048),
        # the same from the optimal basis of the family's base LP, repaired where it is infeasible
        dict(name="family_warm_1024x2048", what="family", warm=True, m=1024, n=2048),
        # thousands of small LPs of uneven sizes in one call
        dict(name="batch_4096", what="batch", count=4096, m_lo=16, m_hi=256),
        # a handful of small LPs: the chip is mostly empty
        dict(name="batch_48", what="batch", count=48, m_lo=16, m_hi=128),
        # the warm-start network on one instance (features -> logits)
        dict(name="net_infer_1", what="infer", m=1024, n=2048, hidden=512, batch=1),
        # training steps of that network, the weights read back at the end
        dict(name="net_train_256", what="train", m=1024, n=2048, hidden=512, batch=256, steps=16),
        # one PRICE on the caller's own buffers
        dict(name="price_4096x8192", what="price", m=4096, n=8192),
    ]


def _span(rng, lo, hi):
    """An integer between lo and hi, even over the logarithm."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.choice(["lp", "lp", "lp", "family", "batch", "infer", "train", "price"])
    if what == "lp":
        family = rng.choice(["int", "real", "degenerate", "general"])
        lo, hi = {"int": (40, 600), "real": (100, 3000), "degenerate": (60, 300), "general": (30, 260)}[family]
        m = _span(rng, lo, hi)
        return dict(what="lp", family=family, m=m, n=rng.randint(m, 2 * m))
    if what == "family":
        m = _span(rng, 200, 1400)
        return dict(what="family", warm=rng.random() < 0.5, m=m, n=rng.randint(m, 2 * m))
    if what == "batch":
        lo = _span(rng, 16, 64)
        return dict(what="batch", count=_span(rng, 16, 4096), m_lo=lo, m_hi=rng.randint(lo, 256))
    if what == "infer":
        m = _span(rng, 100, 1400)
        return dict(what="infer", m=m, n=rng.randint(m, 2 * m), hidden=rng.choice([128, 256, 512]),
                    batch=rng.choice([1, 1, 2, 7, 33, 256]))
    if what == "train":
        m = _span(rng, 100, 1400)
        return dict(what="train", m=m, n=rng.randint(m, 2 * m), hidden=rng.choice([128, 256, 512]),
                    batch=rng.choice([32, 100, 256]), steps=rng.randint(4, 16))
    m = _span(rng, 100, 8000)
    return dict(what="price", m=m, n=rng.randint(m, 2 * m) if m <= 4096 else rng.randint(2000, 4000))


# ---- inputs ----------------------------------------------------------------------------

def _gen(seed, tag=0):
    return torch.Generator(device="cuda").manual_seed(1_000_003 * int(seed) + tag)


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device="cuda", dtype=torch.float64)


def _ints(g, lo, hi, *shape):
    return torch.randint(lo, hi + 1, shape, generator=g, device="cuda").to(torch.float64)


def _problem(family, m, n, seed):
    """max c^T x, A x <= b, x >= 0 on the GPU, drawn as lpgen draws its families."""
    g = _gen(seed)
    if family == "int":
        return _ints(g, 1, 100, m, n), 1000.0 + 9000.0 * _rand(g, m), _ints(g, 1, 100, n)
    if family == "real":
        A = _rand(g, m, n)
        A *= _rand(g, m, n) >= 0.1
        return A, n / 4.0 + (n / 4.0) * _rand(g, m), _rand(g, n)
    if family == "degenerate":
        A = _ints(g, -5, 10, m, n)
        b = 1.0 + 99.0 * _rand(g, m)
        b[torch.randperm(m, generator=g, device="cuda")[: int(0.3 * m)]] = 0.0
        return A, b, _ints(g, 1, 20, n)
    # general: x* in [0, 1)^n is feasible, three rows in ten have a negative right-hand side, the last row bounds x
    neg = (_rand(g, m, 1) < 0.3).to(torch.float64)
    A = torch.floor(-2.0 - 8.0 * neg + _rand(g, m, n) * 13.0)
    A[m - 1] = 1.0
    xs = _rand(g, n)
    b = A @ xs + _rand(g, m)
    b[m - 1] = xs.sum() + n
    return A, b, _ints(g, 1, 20, n)


def _instance(case, seed):
    """One instance of the family of a base LP: every entry of the base times its own N(1, 0.05^2) draw."""
    base = _problem("real", case["m"], case["n"], 77)
    g = _gen(seed, 1)
    return base, tuple(t * (1.0 + 0.05 * torch.randn(t.shape, generator=g, device="cuda", dtype=torch.float64))
                       for t in base)


def _small_lps(case, seed):
    sizes = np.random.default_rng(case["count"])  # the sizes belong to the case, the numbers to the seed
    ms = sizes.integers(case["m_lo"], case["m_hi"] + 1, case["count"])
    ns = ms + sizes.integers(0, ms + 1)
    rng = np.random.default_rng([int(seed), 3])
    at = np.concatenate([[0], np.cumsum(ms * ns)])
    flat = rng.integers(1, 101, int(at[-1]), dtype=np.uint8).astype(np.float64)
    return [(flat[at[k]:at[k + 1]].reshape(int(ms[k]), int(ns[k])), 1000.0 + 9000.0 * rng.random(int(ms[k])),
             rng.integers(1, 101, int(ns[k])).astype(np.float64)) for k in range(case["count"])]


def _net_data(case, seed):
    """Network parameters, and per step a batch of standardised features and 0/1 labels."""
    n_in, hid, n_out = 2 * (case["m"] + case["n"]), case["hidden"], case["m"] + case["n"]
    g = _gen(seed, 2)
    parts = []
    for a, b in ((n_in, hid), (hid, hid), (hid, n_out)):
        lim = math.sqrt(6.0 / a)
        parts.append(((torch.rand(a, b, generator=g, device="cuda") * 2.0 - 1.0) * lim).flatten())
        parts.append(torch.zeros(b, device="cuda"))
    steps = case.get("steps", 1)
    X = torch.randn(steps, case["batch"], n_in, generator=g, device="cuda")
    T = (torch.rand(steps, case["batch"], n_out, generator=g, device="cuda") < 1.0 / 3.0).to(torch.float32)
    return torch.cat(parts).cpu().numpy(), X, T


def _price_data(case, seed):
    """A column by column, costs, and the duals and basis of a solve under way: one row in twelve has a dual."""
    m, n = case["m"], case["n"]
    g = _gen(seed, 4)
    lda = m + (m & 1)
    At = torch.zeros(n, lda, device="cuda", dtype=torch.float64)
    At[:, :m] = _rand(g, n, m)
    At[:, :m] *= _rand(g, n, m) >= 0.1
    live = torch.randperm(m, generator=g, device="cuda")[: max(1, m // 12)]
    y = torch.zeros(m, device="cuda", dtype=torch.float64)
    y[live] = _rand(g, live.numel()) * (2.0 / live.numel())
    pos = torch.full((n + m,), -1, device="cuda", dtype=torch.int32)
    pos[n:] = torch.arange(m, device="cuda", dtype=torch.int32)
    pos[n + live] = -1
    basic = torch.randperm(n, generator=g, device="cuda")[: live.numel()]
    pos[basic] = live[: basic.numel()].to(torch.int32)
    return At, lda, _rand(g, n), y, pos


# ---- one pass ----------------------------------------------------------------------------

def prepare(case, seed):
    what = case["what"]
    if what == "lp":
        return dict(what=what, lp=lpgb.LP(*_problem(case["family"], case["m"], case["n"], seed)))
    if what == "family":
        base, inst = _instance(case, seed)
        s = dict(what=what, lp=lpgb.LP(*base), inst=inst, basis=None)
        if case["warm"]:
            s["lp"].solve()
            s["basis"] = s["lp"].basis()
        return s
    if what == "batch":
        return dict(what=what, batch=lpgb.Batch(_small_lps(case, seed)))
    if what in ("infer", "train"):
        params, X, T = _net_data(case, seed)
        n_in, n_out = X.shape[-1], T.shape[-1]
        net = lpgb.MLP(n_in, case["hidden"], n_out, case["batch"])
        net.set_params(params)
        if what == "infer":
            return dict(what=what, net=net, X=X[0], logits=torch.empty_like(T[0]))
        return dict(what=what, net=net, X=X, T=T)
    At, lda, c, y, pos = _price_data(case, seed)
    return dict(what=what, m=case["m"], n=case["n"], A=At, lda=lda, c=c, y=y, pos=pos,
                q=torch.zeros(1, dtype=torch.int32, device="cuda"),
                dq=torch.zeros(1, dtype=torch.float64, device="cuda"))


def run(s):
    what = s["what"]
    if what == "lp":
        s["lp"].reset()
        res = s["lp"].solve()
        x, y, z = s["lp"].solution()
        return dict(status=res.status, x=x, y=y, z=z)
    if what == "family":
        lp = s["lp"]
        lp.update_problem(*s["inst"])
        if s["basis"] is not None:
            lp.set_basis_repair(s["basis"], lp.m)
        res = lp.solve()
        x, y, z = lp.solution()
        return dict(status=res.status, x=x, y=y, z=z)
    if what == "batch":
        s["batch"].solve()
        status, iters, obj, xs, ys = s["batch"].results()
        return dict(status=status, iters=iters, z=obj, x=np.concatenate(xs), y=np.concatenate(ys))
    if what == "infer":
        s["net"].forward(s["X"], s["logits"])
        return s["logits"]
    if what == "train":
        loss = [s["net"].train_step(x, t, 1e-3) for x, t in zip(s["X"], s["T"])]
        return dict(loss=np.array(loss, np.float32), params=s["net"].get_params())
    rc = lpgb.price_static(s["m"], s["n"], s["A"], s["lda"], s["c"], s["y"], s["pos"], 1e-9, s["q"], s["dq"],
                           torch.cuda.current_stream().cuda_stream)
    if rc != lpgb.LP_OK:
        raise RuntimeError(f"price_static: {rc}")
    return dict(q=s["q"], dq=s["dq"])


def work(case):
    """Inputs read once, outputs written once; of the arithmetic only what is known before the solve: pricing every
    column once, which proves the optimum."""
    m, n, what = case.get("m", 0), case.get("n", 0), case["what"]
    if what in ("lp", "family"):
        return dict(bytes=8.0 * (m * n + 2 * (m + n)), flops=2.0 * m * n)
    if what == "batch":
        mean_m = 0.5 * (case["m_lo"] + case["m_hi"])
        sq = (case["m_hi"] - case["m_lo"]) ** 2 / 12.0 + mean_m ** 2
        return dict(bytes=8.0 * case["count"] * (1.5 * sq + 5.0 * mean_m), flops=3.0 * case["count"] * sq)
    n_in, n_out, h, b = 2 * (m + n), m + n, case.get("hidden", 0), case.get("batch", 0)
    weights = n_in * h + h * h + h * n_out
    if what == "infer":
        return dict(bytes=2.0 * weights + 4.0 * b * (n_in + n_out), flops=2.0 * b * weights)
    if what == "train":
        # the FP32 weights and moments read and written per step, the batch read; forward, and two products per layer
        # but the first in the backward pass
        return dict(bytes=case["steps"] * (24.0 * weights + 4.0 * b * (n_in + n_out)) + 4.0 * weights,
                    flops=case["steps"] * 2.0 * b * (3 * weights - n_in * h))
    return dict(bytes=8.0 * (m * n + m + n) + 4.0 * (m + n) + 12.0, flops=2.0 * m * n)


# ---- the same in 64 bits, by plain torch ---------------------------------------------------

def _pivots(A, b, c, basis, Binv, limit=60000):
    """Dantzig's revised simplex on a stack of LPs (leading dimension) from feasible bases; the bases at the end."""
    L, m, n = A.shape
    rows, eye = torch.arange(L, device=A.device), torch.eye(m, device=A.device, dtype=A.dtype)
    call = torch.cat([c, torch.zeros(L, m, device=A.device, dtype=A.dtype)], 1)
    xb = (Binv @ b[:, :, None])[:, :, 0]
    for it in range(limit):
        if it % 1000 == 999 and L == 1:
            B = torch.cat([A[0], eye], 1)[:, basis[0]]
            Binv = torch.linalg.inv(B)[None]
            xb = (Binv @ b[:, :, None])[:, :, 0]
        y = (torch.gather(call, 1, basis)[:, None, :] @ Binv)[:, 0]
        d = torch.cat([c - (y[:, None, :] @ A)[:, 0], -y], 1)
        d.scatter_(1, basis, -math.inf)
        best, q = d.max(1)
        go = best > 1e-9
        if it % 8 == 0 and not bool(go.any()):
            return basis, Binv
        col = torch.where((q < n)[:, None], A[rows, :, q.clamp(max=n - 1)], eye[(q - n).clamp(min=0)])
        al = (Binv @ col[:, :, None])[:, :, 0]
        ratio = torch.where(al > 1e-9, xb.clamp(min=0.0) / al, math.inf)
        theta = ratio.min(1).values
        tie = torch.where(ratio <= (theta + 1e-12 * theta.clamp(min=1.0))[:, None], al, -math.inf)
        r = tie.max(1).indices
        ar, go = al[rows, r], go & torch.isfinite(theta)
        rho = Binv[rows, r] / ar[:, None]
        al[rows, r] = ar - 1.0
        al = torch.where(go[:, None], al, 0.0)
        rho = torch.where(go[:, None], rho, 0.0)
        theta = torch.where(go, theta, 0.0)
        enters = torch.where(go, theta, xb[rows, r])
        xb = xb - al * theta[:, None]
        xb[rows, r] = enters
        Binv.baddbmm_(al[:, :, None], rho[:, None, :], alpha=-1.0)
        basis[rows, r] = torch.where(go, q, basis[rows, r])
    return None, None


def _vertex(A, b, c, basis):
    """x, y and the objective of one LP at a basis, or None where it is not an optimum."""
    m, n = A.shape
    full = torch.cat([A, torch.eye(m, device=A.device, dtype=A.dtype)], 1)
    cost = torch.cat([c, torch.zeros(m, device=A.device, dtype=A.dtype)])
    lu = torch.linalg.lu_factor(full[:, basis])

    def solve(rhs, adjoint):
        v = torch.linalg.lu_solve(*lu, rhs[:, None], adjoint=adjoint)[:, 0]
        B = full[:, basis].T if adjoint else full[:, basis]
        return v + torch.linalg.lu_solve(*lu, (rhs - B @ v)[:, None], adjoint=adjoint)[:, 0]

    xb, y = solve(b, False), solve(cost[basis], True)
    x = torch.zeros(n + m, device=A.device, dtype=A.dtype).index_put((basis,), xb)[:n]
    scale = float(b.abs().max())
    if float(xb.min()) < -1e-7 * scale or float((c - y @ A).max()) > 1e-7 or float(y.min()) < -1e-7:
        return None
    return x, y, float(c @ x)


def _optimum(A, b, c):
    m, n = A.shape
    eye = torch.eye(m, device=A.device, dtype=A.dtype)
    if float(b.min()) < 0.0:  # one artificial column for the rows with a negative right-hand side
        A1 = torch.cat([A, -(b < 0.0).to(A.dtype)[:, None]], 1)
        c1 = torch.zeros(n + 1, device=A.device, dtype=A.dtype)
        c1[n] = -1.0
        basis = torch.arange(n + 1, n + 1 + m, device=A.device)
        basis[int(b.argmin())] = n
        Binv = torch.linalg.inv(torch.cat([A1, eye], 1)[:, basis])
        basis, Binv = _pivots(A1[None], b[None], c1[None], basis[None], Binv[None].clone())
        if basis is None or bool((basis == n).any()):
            return None
        basis = torch.where(basis > n, basis - 1, basis)
    else:
        basis, Binv = torch.arange(n, n + m, device=A.device)[None], eye[None].clone()
    basis, _ = _pivots(A[None], b[None], c[None], basis, Binv)
    return None if basis is None else _vertex(A, b, c, basis[0])


def _exact_batch(case, seed):
    lps = _small_lps(case, seed)
    M, N = max(p[0].shape[0] for p in lps), max(p[0].shape[1] for p in lps)
    x, y, z = [], [], []
    for k0 in range(0, len(lps), 512):
        part = lps[k0:k0 + 512]
        A, b, c = np.zeros((len(part), M, N)), np.ones((len(part), M)), np.full((len(part), N), -1.0)
        for k, p in enumerate(part):
            A[k, :p[0].shape[0], :p[0].shape[1]], b[k, :len(p[1])], c[k, :len(p[2])] = p
        A, b, c = (torch.from_numpy(t).cuda() for t in (A, b, c))
        Binv = torch.eye(M, device="cuda", dtype=torch.float64).repeat(len(part), 1, 1)
        basis, _ = _pivots(A, b, c, torch.arange(N, N + M, device="cuda").repeat(len(part), 1), Binv)
        if basis is None:
            return None
        cost = torch.cat([c, torch.zeros_like(b)], 1)
        B = torch.gather(torch.cat([A, torch.eye(M, device="cuda", dtype=torch.float64).expand(len(part), M, M)], 2),
                         2, basis[:, None, :].expand(-1, M, -1))
        xb = torch.linalg.solve(B, b[:, :, None])[:, :, 0]
        yy = torch.linalg.solve(B.transpose(1, 2), torch.gather(cost, 1, basis)[:, :, None])[:, :, 0]
        xx = torch.zeros_like(cost).scatter(1, basis, xb)[:, :N].cpu().numpy()
        yy = yy.cpu().numpy()
        for k, p in enumerate(part):
            x.append(xx[k, :p[0].shape[1]])
            y.append(yy[k, :p[0].shape[0]])
            z.append(float(p[2] @ x[-1]))
    return dict(status=None, iters=None, z=np.array(z), x=np.concatenate(x), y=np.concatenate(y))


def _exact_net(case, seed, train):
    params, X, T = _net_data(case, seed)
    h = case["hidden"]
    sizes = [(X.shape[-1], h), (h,), (h, h), (h,), (h, T.shape[-1]), (T.shape[-1],)]
    p = [torch.from_numpy(v).cuda().double().reshape(s) for v, s in
         zip(np.split(params, np.cumsum([int(np.prod(s)) for s in sizes])[:-1]), sizes)]
    m1, m2, losses = [torch.zeros_like(v) for v in p], [torch.zeros_like(v) for v in p], []
    for t in range(case.get("steps", 1)):
        x = X[t].double()
        a1 = torch.relu(x @ p[0] + p[1])
        a2 = torch.relu(a1 @ p[2] + p[3])
        z = a2 @ p[4] + p[5]
        if not train:
            return z
        tt, B = T[t].double(), case["batch"]
        losses.append(float((torch.nn.functional.softplus(z) - tt * z).sum()) / B)
        dz = (torch.sigmoid(z) - tt) / B
        d2 = (dz @ p[4].T) * (a2 > 0)
        d1 = (d2 @ p[2].T) * (a1 > 0)
        for v, u, w, g in zip(p, m1, m2, (x.T @ d1, d1.sum(0), a1.T @ d2, d2.sum(0), a2.T @ dz, dz.sum(0))):
            u.mul_(0.9).add_(g, alpha=0.1)
            w.mul_(0.999).add_(g * g, alpha=0.001)
            v -= 1e-3 * (u / (1 - 0.9 ** (t + 1))) / ((w / (1 - 0.999 ** (t + 1))).sqrt() + 1e-8)
    return dict(loss=np.array(losses), params=torch.cat([v.flatten() for v in p]))


def exact(case, seed):
    what = case["what"]
    if what in ("lp", "family"):
        if what == "family":
            A, b, c = _instance(case, seed)[1]
        else:
            A, b, c = _problem(case["family"], case["m"], case["n"], seed)
        if case.get("family") == "degenerate":  # x = 0 is the only feasible point; the duals are not unique
            return None
        got = _optimum(A, b, c)
        return None if got is None else dict(status=None, x=got[0], y=got[1], z=got[2])
    if what == "batch":
        return _exact_batch(case, seed)
    if what in ("infer", "train"):
        return _exact_net(case, seed, what == "train")
    At, _, c, y, pos = _price_data(case, seed)
    m, n = case["m"], case["n"]
    d = torch.cat([c - At[:, :m] @ y, -y])
    d[pos >= 0] = -math.inf
    return dict(q=None, dq=d.max().reshape(1))
