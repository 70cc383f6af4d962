"""Timed calls of the library's public entry points, with their inputs, work and accuracy.

A case is a dict of plain values: its "kind" names the entry point, the rest its sizes and
options.  listed() gives twelve of them, draw() more of the same ranges; prepare() makes a
case's inputs and the workspace a program keeps, run() is one call, exact() the same
outputs from plain numpy in 64 bits where that takes seconds.
"""
import math

import numpy as np
import torch

import paper_2608_18147_gb300 as E
from paper_2608_18147_gb300 import workloads

# The solves' options as the benchmark uses them: a refinement that ends by its stop rule.
REFINE_ROUNDS, REFINE_TOL = 500, 1e-9
LAMBDA_LO, LAMBDA_HI, SEARCH_ROUNDS = 1e-8, 1e3, 6  # the library's default search


def listed():
    return [
        # Encode of one small tensor (a bias, one attention head's row) with a 3-bit codebook:
        # the cost of the call itself.
        dict(name="encode_4097_m8", kind="encode", d=4097, m=8, dist="normal"),
        # Encode of a large weight matrix or gradient bucket with a 4-bit codebook, ragged length.
        dict(name="encode_67108867_m16", kind="encode", d=67108867, m=16, dist="student_t"),
        # Time-shared encode (two codebooks) of one layer's gradient.
        dict(name="timeshare_encode_16777216_m16", kind="timeshare_encode", d=16777216, m=16, beta=0.563,
             dist="lognormal"),
        # Sort, weighted histogram and prefix sums of one weight matrix: step 1 of every solve.
        dict(name="prepare_4000037", kind="prepare", d=4000037, dist="mixture"),
        # The smallest budgeted solve (search, refinement): launches and latency.
        dict(name="solve_normal_1024_s8", kind="solve", d=1024, s=8, budget=2.0, dist="normal", resident=True,
             refine=True),
        # A gradient-like vector, the ordinary size; budget search without refinement.
        dict(name="solve_lognormal_16384_s16", kind="solve", d=16384, s=16, budget=1.0, dist="lognormal",
             resident=True, refine=False),
        # The largest: the benchmark's own workload, with refinement until its stop rule.
        dict(name="solve_student_t_131072_s16", kind="solve", d=131072, s=16, budget=2.5, dist="student_t",
             resident=True, refine=True),
        # Weight-like values with a 5-bit codebook: the wide codebooks' layout of the DP.
        dict(name="solve_mixture_50001_s32", kind="solve", d=50001, s=32, budget=4.0, dist="mixture",
             resident=True, refine=False),
        # The call with its default flags (no interval-cost table in the workspace), odd length.
        dict(name="solve_default_12289_s16", kind="solve", d=12289, s=16, budget=3.0, dist="normal",
             resident=False, refine=False),
        # One codebook per KV-cache row, head size 128.
        dict(name="rows_8192x128_s8", kind="rows", rows=8192, d=128, s=8, budget=3.0),
        # One codebook per group of a group-wise weight quantizer, groups longer than 128 values.
        dict(name="rows_64x300_s8", kind="rows", rows=64, d=300, s=8, budget=3.0),
        # Codebook values drawn from a uniform grid instead of the input's own values.
        dict(name="grid_1000_d100003_s16", kind="grid", d=100003, n=1000, s=16, budget=2.5, dist="student_t"),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["encode", "encode", "timeshare_encode", "prepare", "solve", "solve", "solve", "rows", "rows",
                       "grid"])
    dist = rng.choice(["normal", "lognormal", "student_t", "mixture"])
    if kind == "encode":
        return dict(kind=kind, d=_log_int(rng, 1000, 1 << 26), m=rng.choice([4, 8, 15, 16, 32]), dist=dist)
    if kind == "timeshare_encode":
        return dict(kind=kind, d=_log_int(rng, 1 << 14, 1 << 24), m=rng.choice([8, 16, 32]),
                    beta=round(rng.uniform(0.05, 0.95), 3), dist=dist)
    if kind == "prepare":
        return dict(kind=kind, d=_log_int(rng, 1 << 10, 1 << 22), dist=dist)
    if kind == "solve":
        s = rng.choice([6, 8, 12, 16, 16, 32])
        resident = rng.random() < 0.7
        return dict(kind=kind, d=_log_int(rng, 300, 32768 if resident else 12288), s=s,
                    budget=rng.choice([1.0, 1.5, 2.0, 2.5]) + (1.0 if s == 32 else 0.0), dist=dist, resident=resident,
                    refine=rng.random() < 0.4)
    if kind == "rows":
        if rng.random() < 0.6:
            return dict(kind=kind, rows=_log_int(rng, 16, 8192), d=rng.randint(32, 128), s=rng.choice([4, 8, 16]),
                        budget=rng.choice([1.5, 2.0, 3.0]))
        return dict(kind=kind, rows=_log_int(rng, 4, 64), d=rng.randint(129, 512), s=rng.choice([4, 8, 16]),
                    budget=rng.choice([1.5, 2.0, 3.0]))
    return dict(kind=kind, d=_log_int(rng, 4096, 131072), n=_log_int(rng, 64, 2048), s=rng.choice([8, 16]),
                budget=rng.choice([1.5, 2.0, 2.5]), dist=dist)


# ------------------------------------------------------------------ inputs

def _vector(dist, d, seed):
    """The workloads' distributions, drawn on the GPU (long vectors) as fp32."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    z = torch.randn(d, generator=g, device="cuda")
    if dist == "normal":
        return z
    if dist == "lognormal":
        u = torch.rand(d, generator=g, device="cuda")
        return torch.where(u < 0.5, -1.0, 1.0) * torch.exp(z)
    if dist == "student_t":  # 1e-3 times Student-t with 3 degrees of freedom
        chi = torch.randn(d, generator=g, device="cuda").square_()
        for _ in range(2):
            chi += torch.randn(d, generator=g, device="cuda").square_()
        return z.div_((chi / 3).sqrt_()).mul_(1e-3)
    u = torch.rand(d, generator=g, device="cuda")
    return torch.where(u < 0.1, 10.0, 1.0) * z


def _repeated(x):
    """d entries with exactly 3 d / 4 distinct values, in random order (quantized or tied weights)."""
    d = x.numel()
    g = torch.Generator(device="cuda").manual_seed(d)
    v = torch.unique(x)
    v = v[torch.randperm(v.numel(), generator=g, device="cuda")[: 3 * d // 4]]
    again = torch.randint(0, v.numel(), (d - v.numel(),), generator=g, device="cuda")
    return torch.cat([v, v[again]])[torch.randperm(d, generator=g, device="cuda")].contiguous()


def _short_vector(case, seed):
    gen = {"normal": workloads.normal, "lognormal": workloads.signed_lognormal, "student_t": workloads.student_t,
           "mixture": workloads.mixture}[case["dist"]]
    return gen(case["d"], seed)


def _codebook(x, m, shift=0.0):
    """m values of x that span it: its ends and, between them, quantiles of a sample."""
    sample = torch.sort(x[:: max(1, x.numel() // 65536)]).values
    at = ((torch.arange(1, m - 1, device="cuda") + shift) / (m - 1) * (sample.numel() - 1)).round().long()
    return torch.unique(torch.cat([x.min().view(1), sample[at], x.max().view(1)]))


def _flags(case):
    return E.RESIDENT_COSTS if case.get("resident") else 0


def prepare(case, seed):
    kind, d = case["kind"], case["d"]
    if kind == "encode":
        x = _vector(case["dist"], d, seed)
        return dict(case=case, x=x, Q=_codebook(x, case["m"]), seed=seed,
                    ws=torch.empty(256, dtype=torch.uint8, device="cuda"))
    if kind == "timeshare_encode":
        x = _vector(case["dist"], d, seed)
        return dict(case=case, x=x, Q=_codebook(x, case["m"] - 1), Qp=_codebook(x, case["m"], 0.3), seed=seed,
                    ws=torch.empty(256, dtype=torch.uint8, device="cuda"))
    if kind == "prepare":
        ws = torch.empty(int(E.lib().ecasq_workspace_size_prep(d)), dtype=torch.uint8, device="cuda")
        return dict(case=case, x=_repeated(_vector(case["dist"], d, seed)), ws=ws)
    if kind == "solve":
        return dict(case=case, x=torch.from_numpy(_short_vector(case, seed)).cuda(),
                    ws=E.workspace(d, case["s"], flags=_flags(case)), Q=torch.zeros(case["s"], device="cuda"))
    if kind == "rows":
        X = torch.from_numpy(workloads.kv_rows(case["rows"], d, seed)).cuda()
        return dict(case=case, X=X, ws=E.workspace(d, case["s"], case["rows"]))
    x = _short_vector(case, seed)
    P = E.uniform_grid(x, case["n"])
    ws = torch.empty(int(E.lib().ecasq_workspace_size_grid(d, P.size, case["s"], 0)), dtype=torch.uint8, device="cuda")
    return dict(case=case, x=torch.from_numpy(x).cuda(), P=torch.from_numpy(P).cuda(), ws=ws,
                Q=torch.zeros(case["s"], device="cuda"))


# --------------------------------------------------------------------- run

def _solved(state, Q, res):
    state["Q"][: res["m"]].copy_(Q)  # into the program's table of codebooks
    return dict(Q=state["Q"], m=res["m"], p=res["p"], lam=res["lambda"], mse=res["mse"], vnmse=res["vnmse"],
                h_surrogate=res["h_surrogate"], h_exact=res["h_exact"], objective=res["objective"],
                evaluated=res["lambdas_evaluated"], rounds=res["refine_rounds"])


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "encode":
        idx, counts, h = E.ecasq_quantize(state["x"], state["Q"], state["seed"], ws=state["ws"])
        return dict(idx=idx, counts=counts, h=h)
    if kind == "timeshare_encode":
        idx, sel, counts, rate = E.ecasq_quantize_timeshare(state["x"], state["Q"], state["Qp"], case["beta"],
                                                            state["seed"], state["seed"] + 1, ws=state["ws"])
        return dict(idx=idx, sel=sel, counts=counts, h=rate)
    if kind == "prepare":
        return E.ecasq_prepare(state["x"], ws=state["ws"])
    if kind == "solve":
        kw = dict(refine_max_rounds=REFINE_ROUNDS, refine_rel_tol=REFINE_TOL) if case["refine"] else {}
        return _solved(state, *E.ecasq_solve(state["x"], case["s"], budget_bits=case["budget"], ws=state["ws"],
                                             flags=_flags(case), **kw))
    if kind == "rows":
        Q, m, res = E.ecasq_solve_batched(state["X"], case["s"], budget_bits=case["budget"], ws=state["ws"])
        return dict(Q=Q, m=m, lam=res.field("lambda"), mse=res.field("mse"), h_surrogate=res.field("h_surrogate"),
                    h_exact=res.field("h_exact"))
    return _solved(state, *E.ecasq_solve_grid(state["x"], state["P"], case["s"], budget_bits=case["budget"],
                                              ws=state["ws"]))


def _search_ops(n, s):
    """Additions and comparisons of the search's 43 multipliers: every candidate k < j of layers 3..s."""
    return 2.0 * (1 + 7 * SEARCH_ROUNDS) * (s - 2) * n * (n - 1) / 2


def work(case):
    kind, d = case["kind"], case["d"]
    if kind == "encode":  # x in; one index per entry out; about 30 integer and fp32 operations per entry
        return dict(bytes=5 * d + 8 * case["m"], flops=30 * d)
    if kind == "timeshare_encode":  # x in; an index and a part per entry out; two draws per entry
        return dict(bytes=6 * d + 16 * case["m"], flops=50 * d)
    if kind == "prepare":  # x in; v, w, N and two double-double sums per value out
        return dict(bytes=4 * d + (4 + 8 + 8 + 32) * d, flops=20 * d)
    if kind == "solve":
        return dict(bytes=4 * d + 4 * case["s"], flops=_search_ops(d, case["s"]))
    if kind == "rows":
        return dict(bytes=case["rows"] * (4 * d + 4 * case["s"]), flops=case["rows"] * _search_ops(d, case["s"]))
    return dict(bytes=4 * d + 4 * case["n"], flops=_search_ops(case["n"], case["s"]))


def tolerance(case):
    # Indices, counts and codebooks are whole decisions and stay the same; metrics are sums of
    # a few binary64 terms.  The low words of the prefix sums are rounding errors of the high
    # ones: both words are compared, so another correct summation shows in the low word only.
    if case["kind"] == "prepare":
        return dict(rel=1e-9, max=1e-6)
    return dict(rel=1e-13, max=1e-12)


# ------------------------------------------------- 64-bit values (plain numpy)

def _h(y):
    y = np.asarray(y, np.float64)
    return np.where(y > 0, -y * np.log2(np.where(y > 0, y, 1.0)), 0.0)


def _split_sums(values, at):
    """Prefix sums of `values` (exact integers times a power of two) at the positions `at`: (hi, lo)."""
    total, run, pos = 0, [], 0
    for t in at:
        total += sum(values[pos:t])
        pos = t
        run.append(total)
    hi = [float(t) for t in run]
    lo = [float(t - int(h)) for t, h in zip(run, hi)]
    return np.array(hi), np.array(lo)


def _exact_prepare(x):
    x = np.sort(x + np.float32(0))
    v, first, w = np.unique(x, return_index=True, return_counts=True)
    at = np.append(first, x.size).tolist()
    mant, ex = np.frexp(x.astype(np.float64))
    low = int(ex.min()) - 24
    ints = [int(q) << int(e - low - 24) for q, e in zip((mant * (1 << 24)).astype(np.int64), ex)]
    out = dict(p=int(v.size), v=v, w=w.astype(np.int64), N=np.array(at, np.int64))
    for key, vals, power in (("S", ints, low), ("S2", [q * q for q in ints], 2 * low)):
        hi, lo = _split_sums(vals, at)
        out[key + "_hi"], out[key + "_lo"] = np.ldexp(hi, power), np.ldexp(lo, power)
    return out


def _draws(seed, d):
    with np.errstate(over="ignore"):
        z = np.uint64(seed) + np.arange(1, d + 1, dtype=np.uint64) * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return (z ^ (z >> np.uint64(31))) >> np.uint64(40)


def _exact_encode(x, Q, seed):
    t = np.searchsorted(Q, x, side="right") - 1
    gap = np.append(np.diff(Q), np.float32(0)).astype(np.float32)
    up = (_draws(seed, x.size).astype(np.float32) * np.float32(2.0 ** -24)) * gap[t] < x - Q[t]
    return (t + up).astype(np.uint8)


def _entropy(counts, total):
    return float(np.sum(_h(counts / total)))


class _Pairs:
    """Interval costs of all pairs k < j of the candidates v (weights w, d entries; sums N, S, S2 up to
    and including each candidate)."""

    def __init__(self, v, w0, N, S, S2, d):
        self.v, self.w0, self.d = np.asarray(v, np.float64), float(w0), d
        N, S, S2, vl = (np.asarray(a, np.longdouble) for a in (N, S, S2, v))
        k, j = np.s_[:, None], np.s_[None, :]
        n, ds, ds2 = N[j] - N[k], S[j] - S[k], S2[j] - S2[k]
        L = np.where(np.triu(np.ones((len(v), len(v)), bool), 1), vl[j] - vl[k], 1)
        self.upper = np.triu(np.ones((len(v), len(v)), bool), 1)
        self.C = ((vl[k] + vl[j]) * ds - ds2 - vl[k] * vl[j] * n).astype(np.float64)
        self.U = ((ds - vl[k] * n) / L).astype(np.float64)
        self.D = ((vl[j] * n - ds) / L).astype(np.float64)
        self.Phi = _h(self.U / d) + _h(self.D / d)
        self.first = _h(self.U[0] / d) + _h((self.D[0] + self.w0) / d)

    def solve(self, s, lamp):
        """Least C + lamp Phi over codebooks of at most s values: indices."""
        W = np.where(self.upper, self.C + lamp * self.Phi, np.inf)
        dp = np.where(self.upper[0], self.C[0] + lamp * self.first, np.inf)
        back, ends = [], [dp[-1]]
        for _ in range(3, s + 1):
            cand = dp[:, None] + W
            arg = np.argmin(cand, axis=0)
            dp = cand[arg, np.arange(len(arg))]
            back.append(arg)
            ends.append(dp[-1])
        i = int(np.argmin(ends))
        a = [len(self.v) - 1]
        for arg in reversed(back[:i]):
            a.append(int(arg[a[-1]]))
        return np.array([0] + a[::-1]) if len(a) else None

    def metrics(self, a):
        U, D = self.U[a[:-1], a[1:]], self.D[a[:-1], a[1:]]
        mse = float(np.sum(self.C[a[:-1], a[1:]]))
        hs = float(self.first[a[1]] + np.sum(self.Phi[a[1:-1], a[2:]]))
        f = np.concatenate([[self.w0], U]) + np.concatenate([D, [0.0]])
        return mse, hs, float(np.sum(_h(f / self.d)))

    def refine(self, a, lamp, budget):
        a, m = a.copy(), len(a)
        J = self._J(a, lamp)
        rounds = 0
        for rounds in range(1, REFINE_ROUNDS + 1):
            J0 = J
            for colour in (0, 1, 2):
                new = a.copy()
                for l in range(3 if colour == 0 else colour, m - 1, 3):
                    lo, hi = a[l - 1], a[l + 1]
                    c = np.arange(lo + 1, hi)
                    left = self.w0 if l == 1 else self.U[a[l - 2], lo]
                    right = 0.0 if l == m - 2 else self.D[hi, a[l + 2]]
                    ent = (_h((left + self.D[lo, c]) / self.d) + _h((self.U[lo, c] + self.D[c, hi]) / self.d) +
                           _h((self.U[c, hi] + right) / self.d))
                    obj = self.C[lo, c] + self.C[c, hi] + lamp * ent
                    if obj.min() < obj[a[l] - lo - 1]:
                        new[l] = c[int(np.argmin(obj))]
                if not np.array_equal(new, a) and self.metrics(new)[2] <= budget:
                    a = new
            J = self._J(a, lamp)
            if not J0 - J > REFINE_TOL * abs(J0):
                break
        return a, rounds

    def _J(self, a, lamp):
        mse, _, hx = self.metrics(a)
        return mse + lamp * hx


def _midpoints(lo, hi):
    t = [0.0] * 7
    t[3] = math.sqrt(lo * hi)
    t[1], t[5] = math.sqrt(lo * t[3]), math.sqrt(t[3] * hi)
    t[0], t[2], t[4], t[6] = math.sqrt(lo * t[1]), math.sqrt(t[1] * t[3]), math.sqrt(t[3] * t[5]), math.sqrt(t[5] * hi)
    return t


def _exact_solve(pairs, norm2, s, budget, refine):
    evals = []

    def at(lam):
        a = pairs.solve(s, lam * norm2)
        evals.append((lam, a) + pairs.metrics(a))
        return evals[-1]

    best = at(0.0)
    if best[3] > budget:
        lo, hi = LAMBDA_LO, LAMBDA_HI
        for _ in range(SEARCH_ROUNDS):
            pts = [at(t) for t in _midpoints(lo, hi)]
            f = next((q for q, e in enumerate(pts) if e[3] <= budget), None)
            if f is None:
                lo = pts[6][0]
            else:
                lo, hi = (pts[f - 1][0] if f else lo), pts[f][0]
        feasible = [e for e in evals if e[3] <= budget]
        best = min(feasible, key=lambda e: (e[2], e[0])) if feasible else at(hi)
        count = len(evals)
    else:
        for t in _midpoints(LAMBDA_LO, LAMBDA_HI):
            at(t)
        count = 8
    lam, a = best[0], best[1]
    rounds = 0
    if refine:
        a, rounds = pairs.refine(a, lam * norm2, budget)
    mse, hs, hx = pairs.metrics(a)
    Q = np.zeros(s, np.float32)
    Q[: len(a)] = pairs.v[a]
    return dict(Q=Q, m=len(a), p=len(pairs.v), lam=lam, mse=mse, vnmse=mse / norm2,
                h_surrogate=hs, h_exact=hx, objective=mse + lam * norm2 * (hx if refine else hs), evaluated=count,
                rounds=rounds)


def _histogram(x, P=None):
    """Candidates and the sums of all entries up to and including each."""
    v, w = np.unique(x + np.float32(0), return_counts=True)
    vl = v.astype(np.longdouble)
    N, S, S2 = np.cumsum(w), np.cumsum(w * vl), np.cumsum(w * vl * vl)
    norm2 = float(S2[-1])
    if P is None:
        return _Pairs(v, w[0], N, S, S2, x.size), norm2
    at = np.searchsorted(v, P, side="right")
    pad = lambda a: np.concatenate([[0], a])[at]  # noqa: E731
    return _Pairs(P, pad(N)[0], pad(N), pad(S), pad(S2), x.size), norm2


def exact(case, seed):
    """run()'s outputs for these inputs; None where they would take too long (large searches, long encodes)."""
    kind, d = case["kind"], case["d"]
    if kind in ("encode", "timeshare_encode", "prepare") and d > 1 << 20:
        return None
    if kind == "solve" and d > 1024 or kind == "grid" and case["n"] > 1024:
        return None
    if kind == "rows" and case["rows"] * d * d > 2 << 20:
        return None
    if kind in ("encode", "timeshare_encode"):
        st = prepare(case, seed)
        x, Q = st["x"].cpu().numpy(), st["Q"].cpu().numpy()
        idx = _exact_encode(x, Q, seed)
        if kind == "encode":
            counts = np.bincount(idx, minlength=Q.size)
            return dict(idx=idx, counts=counts.astype(np.int32), h=_entropy(counts, d))
        Qp = st["Qp"].cpu().numpy()
        sel = _draws(seed + 1, d) * 2.0 ** -24 < case["beta"]
        idx = np.where(sel, _exact_encode(x, Qp, seed), idx)
        cm, cp = np.bincount(idx[~sel], minlength=Q.size), np.bincount(idx[sel], minlength=Qp.size)
        rate = sum(c.sum() / d * _entropy(c, c.sum()) for c in (cm, cp) if c.sum())
        return dict(idx=idx, sel=sel.astype(np.uint8), counts=np.concatenate([cm, cp]).astype(np.int32), h=float(rate))
    if kind == "prepare":
        return _exact_prepare(_repeated(_vector(case["dist"], d, seed)).cpu().numpy())
    if kind == "solve":
        pairs, norm2 = _histogram(_short_vector(case, seed))
        return _exact_solve(pairs, norm2, case["s"], case["budget"], case["refine"])
    if kind == "grid":
        x = _short_vector(case, seed)
        pairs, norm2 = _histogram(x, E.uniform_grid(x, case["n"]))
        return _exact_solve(pairs, norm2, case["s"], case["budget"], False)
    X = workloads.kv_rows(case["rows"], d, seed)
    Q, out = np.zeros((case["rows"], case["s"]), np.float32), []
    for r, x in enumerate(X):
        pairs, norm2 = _histogram(x)
        out.append(_exact_solve(pairs, norm2, case["s"], case["budget"], False))
        Q[r] = out[-1]["Q"]
    col = lambda k: np.array([o[k] for o in out])  # noqa: E731
    return dict(Q=Q, m=col("m").astype(np.int32), lam=col("lam"), mse=col("mse"), h_surrogate=col("h_surrogate"),
                h_exact=col("h_exact"))
