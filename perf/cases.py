"""The performance cases of the library: what its users have it do, over the sizes they do it at.

A case is a dict of plain values; ``kind`` says which public entry point it goes
through and the other fields are its sizes and options.  Sizes come from the
workloads of ``synth``, the benchmark and the tests.  Inputs are made on the GPU
from the seed alone by the generators' recipes (rows around mixture centres, or
isotropic rows, with log-normal norms; queries drawn from the items or fresh).
"""

import math

import numpy as np
import torch

import paper_2504_13446_gb300 as rkr

TAU, OMEGA, S = 500, 10, 100     # the benchmark's table: tau = 500, 10 buckets of 100 samples


def listed():
    return [
        # One query of a small catalogue through the captured serving session: the
        # smallest call there is, all launches and copies.
        dict(name="session_small", kind="session", n=2000, m=5000, d=32, k=10, tau=TAU, omega=OMEGA,
             s=S, c=2.0, mixture=False),
        # One query against the benchmark's million users through the session: an
        # online recommendation request, bound by the pass over the users.
        dict(name="session_million", kind="session", n=1_000_000, m=100_000, d=200, k=50, tau=TAU,
             omega=OMEGA, s=S, c=2.0, mixture=True),
        # A handful of queries answered one at a time, odd dimension and ragged sizes
        # (rows that are not a multiple of 16 bytes).
        dict(name="single_ragged", kind="single", n=150_001, m=20_011, d=101, nq=8, k=50, tau=TAU,
             omega=OMEGA, s=S, c=2.0, mixture=True),
        # A small catalogue with ragged sizes, approximate and exact batches of a few
        # queries: launches, synchronisations and allocations count.
        dict(name="small_ragged", kind="both", n=12_345, m=3_777, d=37, nq=33, k=7, tau=64, omega=7,
             s=40, c=1.5, mixture=True),
        # The benchmark's c-approximate batch: 10,000 queries from the items against a
        # million users, k in {10, 50, 100}.
        dict(name="approx_batch", kind="approx", n=1_000_000, m=100_000, d=200, nq=10_000, k=0,
             tau=TAU, omega=OMEGA, s=S, c=2.0, mixture=True),
        # The exact batch of the tests at full size: isotropic users, half of the
        # queries fresh (not items), k = 100.
        dict(name="exact_fresh", kind="exact", n=500_000, m=20_000, d=100, nq=1024, k=100, tau=TAU,
             omega=OMEGA, s=S, mixture=False, fresh=0.5),
        # The benchmark's exact batch with half of its users: 10,000 queries from the
        # items, k in {10, 50, 100}.
        dict(name="exact_batch", kind="exact", n=500_000, m=100_000, d=200, nq=10_000, k=0, tau=TAU,
             omega=OMEGA, s=S, mixture=True, fresh=0.0),
        # A small catalogue rebuilt with its exact tables and queried once, as a
        # periodic refresh does it.
        dict(name="rebuild_small", kind="build", n=20_000, m=10_007, d=64, nq=256, k=20, tau=200,
             omega=OMEGA, s=50, c=2.0, mixture=True),
        # The benchmark's step: the index of a million users built with its exact
        # tables, then the approximate and the exact batch of 10,000 queries.
        dict(name="build_and_query", kind="build", n=1_000_000, m=100_000, d=200, nq=10_000, k=0,
             tau=TAU, omega=OMEGA, s=S, c=2.0, mixture=True),
        # The uneven workload scaled down: a bitmap of eligible users per query, k
        # log-uniform up to 1,000, fresh queries, deep count grid; exact and approximate.
        dict(name="uneven_subsets", kind="uneven", n=200_000, m=100_000, d=128, nq=512, kmax=1000,
             tau=TAU, omega=OMEGA, s=S, c=2.0),
        # Exact ranks of given (user, query) pairs: training targets of the learned
        # pruner and quality checks; most pairs lie below the tail lists.
        dict(name="rank_pairs", kind="pairs", n=100_000, m=50_000, d=200, nq=1000, pairs=200_000,
             tau=TAU, omega=OMEGA, s=S, mixture=True),
        # The learned pruner's predictions, and the loss and gradients of one batch.
        dict(name="pruner_step", kind="pruner", batch=65_536, features=65, hidden=256),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["session", "single", "both", "approx", "exact", "build", "uneven", "pairs",
                       "pruner"])
    if kind == "pruner":
        return dict(kind=kind, batch=_log(rng, 1000, 65_536), features=65,
                    hidden=rng.choice([64, 128, 200, 256]))
    d = rng.choice([16, 32, 37, 50, 64, 96, 100, 101, 128, 150, 160, 200])
    table = dict(tau=rng.choice([100, 200, 500]), omega=OMEGA, s=rng.choice([50, 100]))
    c = rng.choice([1.5, 2.0, 3.0])
    mix = rng.random() < 0.7
    if kind == "session":
        return dict(kind=kind, n=_log(rng, 2000, 1_000_000), m=_log(rng, 3000, 100_000), d=d,
                    k=_log(rng, 1, 100), c=c, mixture=mix, **table)
    if kind == "single":
        return dict(kind=kind, n=_log(rng, 2000, 300_000), m=_log(rng, 3000, 50_000), d=d,
                    nq=_log(rng, 1, 16), k=_log(rng, 1, 200), c=c, mixture=mix, **table)
    if kind == "both":
        return dict(kind=kind, n=_log(rng, 2000, 30_000), m=_log(rng, 1000, 10_000), d=d,
                    nq=_log(rng, 4, 128), k=_log(rng, 1, 50), c=c, mixture=mix, **table)
    if kind == "approx":
        return dict(kind=kind, n=_log(rng, 20_000, 1_000_000), m=_log(rng, 5000, 100_000), d=d,
                    nq=_log(rng, 100, 10_000), k=0, c=c, mixture=mix, **table)
    if kind == "exact":
        return dict(kind=kind, n=_log(rng, 20_000, 500_000), m=_log(rng, 5000, 100_000), d=d,
                    nq=_log(rng, 100, 10_000), k=0, mixture=mix, fresh=rng.choice([0.0, 0.5]),
                    **table)
    if kind == "build":
        return dict(kind=kind, n=_log(rng, 20_000, 1_000_000), m=_log(rng, 5000, 100_000), d=d,
                    nq=_log(rng, 100, 10_000), k=0, c=c, mixture=mix, **table)
    if kind == "uneven":
        return dict(kind=kind, n=_log(rng, 50_000, 200_000), m=_log(rng, 20_000, 100_000),
                    d=rng.choice([64, 100, 128]), nq=_log(rng, 64, 512), kmax=1000, c=c, **table)
    return dict(kind=kind, n=_log(rng, 20_000, 100_000), m=_log(rng, 5000, 50_000), d=d,
                nq=_log(rng, 100, 1000), pairs=_log(rng, 10_000, 200_000), mixture=mix, **table)


# ------------------------------------------------------------------ inputs

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(1_000_003 * int(seed) + 17)
    return g


def _rows(g, count, d, centers, sigma):
    """Rows of unit direction (around a random centre, or isotropic) and log-normal norm."""
    x = torch.randn(count, d, generator=g, device="cuda")
    if centers is not None:
        which = torch.randint(0, centers.shape[0], (count,), generator=g, device="cuda")
        x.mul_(0.3 / math.sqrt(d)).add_(centers[which])
    x /= x.norm(dim=1, keepdim=True)
    x *= torch.exp(sigma * torch.randn(count, 1, generator=g, device="cuda"))
    return x


def _sample_positions(seed, m, omega, s):
    """Sample positions inside each bucket of the norm-sorted items, without replacement."""
    rng = np.random.default_rng([int(seed), 7])
    out = np.full((omega, s), -1, np.int32)
    for b in range(omega):
        size = m // omega + (1 if b < m % omega else 0)
        out[b, :min(size, s)] = (np.arange(size) if size <= s
                                 else rng.choice(size, s, replace=False))
    return out


def _inputs(case, seed):
    """U, P, Q on the GPU, k per query on the host, and the table's sample positions."""
    g = _gen(seed)
    n, m, d = case["n"], case["m"], case["d"]
    uneven = case["kind"] == "uneven"
    mixture = case.get("mixture", True)
    sigma = 0.5 if mixture else 0.7
    ncent = 1024 if uneven else 256
    centers = (torch.randn(ncent, d, generator=g, device="cuda") / math.sqrt(d)
               if mixture else None)
    U = _rows(g, n, d, centers, sigma)
    P = _rows(g, m, d, centers, sigma)
    nq = case.get("nq", 1)
    fresh = nq if uneven else int(nq * case.get("fresh", 0.0))
    own = P[torch.randperm(m, generator=g, device="cuda")[:nq - fresh]]
    if own.shape[0] < nq - fresh:            # more queries than items: some items again
        own = torch.cat([own, P[torch.randint(0, m, (nq - fresh - own.shape[0],), generator=g,
                                              device="cuda")]])
    Q = torch.cat([own, _rows(g, fresh, d, centers, sigma)]).contiguous()
    rng = np.random.default_rng([n, nq])     # the same k for every seed: same output sizes
    if uneven:
        k = np.clip(np.rint(np.exp(rng.uniform(0.0, math.log(case["kmax"]), nq))), 1, case["kmax"])
    elif case.get("k", 0):
        k = np.full(nq, case["k"])
    else:
        k = rng.choice([10, 50, 100], nq)
    pos = _sample_positions(seed, m, case["omega"], case["s"])
    return U, P, Q, np.minimum(k, n).astype(np.int32), pos


def _bitmaps(nq, n, seed):
    """Each query's eligible users: 10 % to 100 % of the blocks of 1,024 users."""
    rng = np.random.default_rng([int(seed), 11])
    words = (n + 31) // 32
    blocks = (n + 1023) // 1024
    keep = rng.random((nq, blocks)) < rng.uniform(0.1, 1.0, (nq, 1))
    keep[np.arange(nq), rng.integers(0, blocks - 1, nq)] = True    # one full block at least
    bits = np.repeat(np.where(keep, 0xFFFFFFFF, 0).astype(np.uint32), 32, axis=1)[:, :words]
    if n % 32:
        bits[:, -1] &= np.uint32((1 << (n % 32)) - 1)
    return torch.from_numpy(np.ascontiguousarray(bits).view(np.int32)).cuda()


def _pruner_inputs(case, seed):
    rng = np.random.default_rng(int(seed))
    B, F = case["batch"], case["features"]
    X = rng.standard_normal((B, F), dtype=np.float32) * np.float32(1.0 / math.sqrt(F))
    t = rng.standard_normal(B, dtype=np.float32)
    target = (8.0 - 2.0 * t + 0.5 * rng.standard_normal(B)).astype(np.float32)
    # the network's weights, in the flat order W1, A, b1, V2, b2, v3, b3
    H = case["hidden"]
    params = np.concatenate([
        rng.standard_normal(H * F) / math.sqrt(F), -1.0 + 0.1 * rng.standard_normal(H), np.zeros(H),
        math.log(math.expm1(1.0 / H)) + 0.1 * rng.standard_normal(H * H), np.zeros(H),
        np.full(H, math.log(math.expm1(1.0 / math.sqrt(H)))), np.zeros(1)]).astype(np.float32)
    return X, t, target, params


def prepare(case, seed):
    kind = case["kind"]
    if kind == "pruner":
        X, t, target, params = _pruner_inputs(case, seed)
        pruner = rkr.Pruner(case["features"], case["hidden"])
        pruner.set_params(params)
        return dict(case=case, X=X, t=t, target=target, pruner=pruner)
    U, P, Q, k, pos = _inputs(case, seed)
    st = dict(case=case, Q=Q, k=k, pos=pos)
    if kind == "build":
        st.update(U=U, P=P)
        return st
    exact = {"both": 1, "exact": 1, "uneven": 2, "pairs": 1}.get(kind, 0)
    st["index"] = rkr.Index(U, P, tau=case["tau"], omega=case["omega"], s=case["s"],
                            exact_table=exact, sample_pos=pos)
    if kind == "session":
        st["session"] = rkr.Session(st["index"], case["k"], case["c"])
        st["q"] = Q[0].cpu().numpy()     # a request arrives in host memory
    elif kind == "uneven":
        st["member"] = _bitmaps(len(k), case["n"], seed)
    elif kind == "pairs":
        rng = np.random.default_rng([int(seed), 13])
        st["pair_user"] = rng.integers(0, case["n"], case["pairs"]).astype(np.int32)
        st["pair_query"] = rng.integers(0, len(k), case["pairs"]).astype(np.int32)
    return st


# --------------------------------------------------------------------- run

def _approx(r):
    return {f: r[f] for f in ("users", "n_low", "n_up", "est", "case", "nc")}


def _exact(r):
    return {"users": r[0], "ranks": r[1]}


def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind == "session":
        return _approx(state["session"].query(state["q"], case["k"]))
    if kind == "single":
        return _approx(state["index"].query_approx(state["Q"], state["k"], case["c"], single=True))
    if kind == "approx":
        return _approx(state["index"].query_approx(state["Q"], state["k"], case["c"]))
    if kind == "exact":
        return _exact(state["index"].query_exact(state["Q"], state["k"]))
    if kind == "both":
        return [_approx(state["index"].query_approx(state["Q"], state["k"], case["c"])),
                _exact(state["index"].query_exact(state["Q"], state["k"]))]
    if kind == "uneven":
        args = dict(member=state["member"])
        return [_approx(state["index"].query_approx(state["Q"], state["k"], case["c"], **args)),
                _exact(state["index"].query_exact(state["Q"], state["k"], **args))]
    if kind == "pairs":
        return state["index"].rank_pairs(state["Q"], state["pair_user"], state["pair_query"])
    if kind == "build":
        with rkr.Index(state["U"], state["P"], tau=case["tau"], omega=case["omega"], s=case["s"],
                       exact_table=1, sample_pos=state["pos"]) as idx:
            return [_approx(idx.query_approx(state["Q"], state["k"], case["c"])),
                    _exact(idx.query_exact(state["Q"], state["k"]))]
    y = state["pruner"].forward(state["X"], state["t"])
    loss, grads = state["pruner"].loss_grads(state["X"], state["t"], state["target"])
    return [y, np.float32(loss), grads]


# -------------------------------------------------------------------- work

def work(case):
    """One pass's inputs and outputs, each once, and one inner product of length d per
    (user, query) pair, per (user, item) pair where the index is built, and per item of
    a pair whose rank is asked for."""
    kind = case["kind"]
    if kind == "pruner":
        B, F, H = case["batch"], case["features"], case["hidden"]
        params = H * F + H * H + 4 * H + 1
        return {"bytes": 4.0 * (B * (F + 3) + 2 * params), "flops": 4.0 * 2.0 * B * (F * H + H * H)}
    n, m, d, nq = case["n"], case["m"], case["d"], case.get("nq", 1)
    ksum = nq * (case.get("k", 0) or 53)
    if kind == "session":
        nq, ksum = 1, case["k"]
    if kind == "uneven":
        ksum = nq * (case["kmax"] / math.log(case["kmax"]))
    calls = 2 if kind in ("both", "build", "uneven") else 1
    out = ksum * ({"exact": 8, "pairs": 0}.get(kind, 20) + (8 if calls == 2 else 0))
    flops = 2.0 * n * nq * d * calls
    nbytes = 4.0 * n * d + 4.0 * nq * d + out
    if kind == "single":          # one query at a time
        nbytes += (nq - 1) * 4.0 * n * d
    if kind == "uneven":
        nbytes += nq * n / 8
    if kind == "build":
        flops += 2.0 * n * m * d
        nbytes += 4.0 * m * d
    if kind == "pairs":
        flops = 2.0 * case["pairs"] * m * d
        nbytes = 4.0 * (n + m + nq) * d + 12.0 * case["pairs"]
    return {"bytes": float(nbytes), "flops": float(flops)}


# ------------------------------------------------- the same in 64 bits, plainly

def _scores64(A, X):
    """A X^T, summed left to right in FP64."""
    A, X = A.double(), X.double()
    acc = torch.zeros(A.shape[0], X.shape[0], dtype=torch.float64, device=A.device)
    for i in range(A.shape[1]):
        acc.addcmul_(A[:, i:i + 1], X[:, i].unsqueeze(0))
    return acc


def _order(*keys):
    """Indices sorted by the keys in turn, the index last."""
    o = torch.arange(keys[0].shape[0], device=keys[0].device)
    for key in reversed(keys):
        o = o[torch.sort(key[o], stable=True).indices]
    return o


def _approx64(U, P, Q, k, c, tau, omega, s, pos):
    """Section 4.3's estimates in FP64: one array over all queries, in answer order."""
    n, m = U.shape[0], P.shape[0]
    P64 = P.double()
    norm2 = torch.zeros(m, dtype=torch.float64, device=U.device)
    for i in range(P.shape[1]):
        norm2.addcmul_(P64[:, i], P64[:, i])
    perm = _order(-norm2.sqrt())
    rows, weights, start = [], [], 0
    for b in range(omega):
        size = m // omega + (1 if b < m % omega else 0)
        p = torch.from_numpy(pos[b][pos[b] >= 0].astype(np.int64)).to(U.device)
        rows.append(perm[start + p])
        weights.append(torch.full((p.numel(),), float(s if size <= s else size),
                                  dtype=torch.float64, device=U.device))
        start += size
    X, w = P[torch.cat(rows)], torch.cat(weights)
    lo, step, N = [], [], []
    for a in range(0, n, max(1, (1 << 27) // m)):
        Uc = U[a:a + max(1, (1 << 27) // m)]
        sc = _scores64(Uc, P)
        lo.append(sc.min(dim=1).values)
        step.append((sc.max(dim=1).values - lo[-1]) / (tau - 1))
        del sc
        t = lo[-1][:, None] + torch.arange(tau, dtype=torch.float64, device=U.device) * step[-1][:, None]
        col = torch.searchsorted(t, _scores64(Uc, X), right=False)
        W = torch.zeros(Uc.shape[0], tau + 1, dtype=torch.float64, device=U.device)
        W.scatter_add_(1, col, w.expand(Uc.shape[0], -1).contiguous())
        N.append(W.flip(1).cumsum(1).flip(1)[:, 1:])
    lo, step, N = torch.cat(lo), torch.cat(step), torch.cat(N)
    t = lo[:, None] + torch.arange(tau, dtype=torch.float64, device=U.device) * step[:, None]
    out, top = [], float(m * s)
    for q in range(Q.shape[0]):
        kq = int(k[q])
        uq = _scores64(U, Q[q:q + 1])
        j = torch.searchsorted(t, uq, right=True)[:, 0]
        uq = uq[:, 0]
        at = torch.arange(n, device=U.device)
        nlo = torch.where(j < tau, N[at, j.clamp(max=tau - 1)], torch.zeros_like(uq))
        nup = torch.where(j >= 1, N[at, (j - 1).clamp(min=0)], torch.full_like(uq, top))
        rup, rlow = 1 + nup / s, 1 + nlo / s
        inside = (j >= 1) & (j <= tau - 1)
        t0, t1 = t[at, (j - 1).clamp(min=0)], t[at, j.clamp(max=tau - 1)]
        frac = torch.where(inside, (uq - t0) / torch.where(inside, t1 - t0, torch.ones_like(t0)),
                           torch.zeros_like(uq))
        est = rup - (rup - rlow) * frac
        Rlo, Rup = nlo.sort().values[kq - 1], nup.sort().values[kq - 1]
        if c * (s + Rlo) >= s + Rup:
            pick = _order(nup, nlo)[:kq]
        else:
            sure = s + nup <= c * (s + Rlo)
            first = torch.nonzero(sure)[:, 0]
            first = first[_order(nup[first], nlo[first])]
            rest = torch.nonzero((nlo <= Rup) & ~sure)[:, 0]
            rest = rest[_order(est[rest])][:kq - first.numel()]
            pick = torch.cat([first, rest])
        out.append(est[pick])
    return torch.cat(out).cpu().numpy()


def _pruner64(case, seed):
    """Predictions, loss and gradients of the pruner's network by FP64 autograd."""
    X, t, target, flat = (torch.from_numpy(a).double().cuda() for a in _pruner_inputs(case, seed))
    F, H = case["features"], case["hidden"]
    flat.requires_grad_()
    sizes = [H * F, H, H, H * H, H, H, 1]
    W1, A, b1, V2, b2, v3, b3 = torch.split(flat, sizes)
    sp = torch.nn.functional.softplus
    h1 = torch.relu(X @ W1.view(H, F).T - sp(A) * t[:, None] + b1)
    y = torch.relu(h1 @ sp(V2).view(H, H).T + b2) @ sp(v3) + b3
    loss = 0.5 * ((y - target) ** 2).mean()
    loss.backward()
    return [y.detach().cpu().numpy(), float(loss), flat.grad.cpu().numpy()]


def exact(case, seed):
    kind = case["kind"]
    if kind == "pruner":
        return _pruner64(case, seed)
    if kind in ("exact", "pairs", "uneven"):
        return None
    if float(case["n"]) * (case["m"] + 100 * case.get("nq", 1)) * case["d"] > 6e11:
        return None      # the plain scan of every (user, item) pair would take too long
    U, P, Q, k, pos = _inputs(case, seed)
    est = _approx64(U, P, Q, k, case["c"], case["tau"], case["omega"], case["s"], pos)
    approx = dict(users=None, n_low=None, n_up=None, est=est, case=None, nc=None)
    return [approx, dict(users=None, ranks=None)] if kind in ("both", "build") else approx
