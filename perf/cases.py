"""Performance cases of the multilevel Monte Carlo engine, through its public entry points.

A case is a dict of plain values.  Its "kind" names the call a user makes:

plain     the host-output level call, mlmc_level_sums_ex, once per level 0..level at N samples each:
          the fixed-N_l multilevel estimate, where latency and launches count
level     one level range queued on a stream with device outputs, mlmc_level_sums_async, as the
          precision sweep and callers with their own driver run it (every precision, scheme,
          estimator and payoff; optionally with every sample's Y)
estimate  mlmc_estimate, one adaptive estimate to accuracy eps
batch     mlmc_estimate_batch, a book of options valued together
cv        the learned control variate's two estimators on one level, mlmc_cv_level_sums and
          mlmc_cv_mean_sums, with installed parameters
grad      mlmc_mlp_grad, loss and gradient of the control variate's network on one batch of rows

The option is the benchmark's: GBM with S0 = K = 100, r = 0.05, sigma = 0.2, T = 1; the seed of a
case is the seed of its random numbers (batches draw their options from it as well).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1505_00965_gb300 import mlmc, workloads

S0, K, R, SIGMA, T = 100.0, 100.0, 0.05, 0.2, 1.0


def listed():
    return [
        # the plain FP64 workload: European call, levels 0..4, 10^4 samples each; the smallest calls
        {"name": "plain64_european_l0to4", "kind": "plain", "precision": "fp64", "payoff": "european", "M": 4,
         "level": 4, "N": 10_000},
        # the precision sweep at its 10^7 samples: the digital call of the FP32 stream in FP64 ...
        {"name": "sweep64_digital_l2", "kind": "level", "precision": "fp64_stream32", "payoff": "digital", "M": 4,
         "level": 2, "N": 10_000_000, "first": 0, "scheme": "em", "estimator": "coupled", "per_sample": False},
        # ... and the Asian call on a deeper level (fewer samples there, as the sweep takes)
        {"name": "sweep64_asian_l5", "kind": "level", "precision": "fp64", "payoff": "asian", "M": 4, "level": 5,
         "N": 300_007, "first": 0, "scheme": "em", "estimator": "coupled", "per_sample": False},
        # a deep lookback level over a ragged number of whole-path samples
        {"name": "lookback32_l6", "kind": "level", "precision": "fp32", "payoff": "lookback", "M": 4, "level": 6,
         "N": 1_000_003, "first": 0, "scheme": "em", "estimator": "coupled", "per_sample": False},
        # the deepest level of the benchmark with few samples: paths split over lanes, latency bound
        {"name": "asian32_l8_few", "kind": "level", "precision": "fp32", "payoff": "asian", "M": 4, "level": 8,
         "N": 1003, "first": 12_345, "scheme": "em", "estimator": "coupled", "per_sample": False},
        # Milstein with antithetic pairs, every sample's Y kept (a caller with its own statistics)
        {"name": "asian32_milstein_anti_l4", "kind": "level", "precision": "fp32", "payoff": "asian", "M": 4,
         "level": 4, "N": 1_000_000, "first": 0, "scheme": "milstein", "estimator": "antithetic",
         "per_sample": True},
        # the headline: time to eps = 1e-3 for the Asian call, FP32 paths
        {"name": "estimate32_asian_1e-3", "kind": "estimate", "precision": "fp32", "payoff": "asian", "eps": 1e-3,
         "scheme": "em", "estimator": "coupled"},
        # the benchmark's other option, whose rounds run to the deepest level
        {"name": "estimate32_lookback_1e-3", "kind": "estimate", "precision": "fp32", "payoff": "lookback",
         "eps": 1e-3, "scheme": "em", "estimator": "coupled"},
        # plain FP64 multilevel Monte Carlo, the form the FP32 one is quoted against
        {"name": "estimate64_asian_1e-3", "kind": "estimate", "precision": "fp64", "payoff": "asian", "eps": 1e-3,
         "scheme": "em", "estimator": "coupled"},
        # a book of options of uneven cost in one call
        {"name": "batch32_96", "kind": "batch", "n": 96, "eps_lo": 2e-3, "eps_hi": 1e-2},
        # the learned control variate on the deepest level that uses it
        {"name": "cv_asian_l2", "kind": "cv", "payoff": "asian", "level": 2, "N": 4_000_000, "replicates": 128},
        # the training direction: loss and gradient of one large batch
        {"name": "cv_grad_65536", "kind": "grad", "rows": 65_536},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choices(["level", "plain", "estimate", "batch", "cv", "grad"], [60, 8, 14, 6, 8, 4])[0]
    if kind in ("level", "plain"):
        precision = rng.choices(["fp32", "fp64", "fp64_stream32"], [50, 25, 25])[0]
        payoff = rng.choice(["european", "asian", "lookback", "digital"])
        M = rng.choices([4, 2, 8], [70, 20, 10])[0]
        level = rng.randint(0, {4: 8, 2: 13, 8: 5}[M])
        if kind == "plain":
            return {"kind": kind, "precision": precision, "payoff": payoff, "M": M, "level": min(level, 5),
                    "N": int(_log(rng, 1e2, 1e5)) | 1}
        steps = _log(rng, 1e4, 4e9 if precision == "fp32" else 3e8)
        N = max(1, int(steps / M ** level)) | rng.randint(0, 1)
        if payoff == "digital" and N < 20_000:
            payoff = "european"  # a few digital differences are all zero
        return {"kind": kind, "precision": precision, "payoff": payoff, "M": M, "level": level, "N": N,
                "first": rng.choice([0, rng.randint(1, 10 ** 9)]), "scheme": rng.choices(["em", "milstein"], [3, 1])[0],
                "estimator": rng.choices(["coupled", "single", "antithetic" if M < 8 else "coupled"], [6, 1, 2])[0],
                "per_sample": N <= 2_000_000 and rng.random() < 0.25}
    if kind == "estimate":
        precision = rng.choices(["fp32", "fp64"], [2, 1])[0]
        payoff = rng.choice(["european", "asian", "lookback", "digital"])
        lo = {"fp32": 1e-3, "fp64": 1e-3 if payoff in ("european", "asian") else 4e-3}[precision]
        return {"kind": kind, "precision": precision, "payoff": payoff, "eps": round(_log(rng, lo, 1e-2), 6),
                "scheme": rng.choices(["em", "milstein"], [3, 1])[0],
                "estimator": rng.choices(["coupled", "antithetic"], [3, 1])[0]}
    if kind == "batch":
        return {"kind": kind, "n": int(_log(rng, 8, 96)), "eps_lo": round(_log(rng, 2e-3, 5e-3), 6), "eps_hi": 1e-2}
    if kind == "cv":
        return {"kind": kind, "payoff": rng.choice(["asian", "european", "lookback"]), "level": rng.randint(0, 3),
                "N": int(_log(rng, 1e4, 4e6)) | 1, "replicates": int(_log(rng, 8, 128))}
    return {"kind": kind, "rows": 32 * int(_log(rng, 8, 2048))}


# ------------------------------------------------------------------ inputs and calls

def _problem(case):
    return mlmc.Problem(S0=S0, r=R, sigma=SIGMA, T=T, K=K, payoff=case["payoff"], scheme=case.get("scheme", "em"),
                        estimator=case.get("estimator", "coupled"))


def _network(seed):
    """Seeded network parameters of a trained network's size: weights uniform in +-1/sqrt(fan-in),
    small biases, the last layer scaled to the payoff (numpy, FP32)."""
    rng = np.random.default_rng(seed)
    w1 = rng.uniform(-1, 1, 64 * 16) / math.sqrt(16)
    b1 = 0.1 * rng.uniform(-1, 1, 64)
    w2 = rng.uniform(-1, 1, 64 * 64) / math.sqrt(64)
    b2 = 0.1 * rng.uniform(-1, 1, 64)
    w3 = 10.0 * rng.uniform(-1, 1, 64) / math.sqrt(64)
    return np.concatenate([w1, b1, w2, b2, w3, [0.5]]).astype(np.float32)


def _rows(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    X = torch.randn(case["rows"], 16, generator=g, device="cuda")
    Y = X[:, 0] + 0.1 * torch.randn(case["rows"], generator=g, device="cuda")
    return X, Y


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case, "seed": seed, "kind": kind}
    if kind in ("level", "plain", "estimate"):
        s["problem"] = _problem(case)
    if kind == "level":
        s["bytes"] = mlmc.mlmc_level_workspace_bytes(case["level"], case["M"], case["N"], case["precision"])
        s["ws"] = torch.zeros(s["bytes"], dtype=torch.uint8, device="cuda")
        s["sums"] = torch.zeros(4, dtype=torch.float64, device="cuda")
        s["y"] = torch.zeros(case["N"], dtype=torch.float64, device="cuda") if case["per_sample"] else None
    elif kind == "batch":
        s["problems"] = workloads.batch_problems(case["n"], seed, (case["eps_lo"], case["eps_hi"]))
        for q in s["problems"]:
            q["seed"] += 1000 * seed
    elif kind == "cv":
        s["cv"] = mlmc.mlmc_cv_create(4, _problem(case))
        mlmc.mlmc_cv_set_params(s["cv"], case["level"], _network(seed))
        s["sums"] = torch.zeros(8, dtype=torch.float64, device="cuda")
        s["mean"] = torch.zeros(2, dtype=torch.float64, device="cuda")
        s["r"] = torch.zeros(case["N"], dtype=torch.float32, device="cuda")
    elif kind == "grad":
        s["params"] = _network(seed)
        s["X"], s["Y"] = _rows(case, seed)
    return s


def _estimate_outputs(ests):
    top = mlmc.MLMC_MAX_LEVELS

    def pad(v, kind):
        return np.array([list(v(e)) + [0] * (top - len(v(e))) for e in ests], dtype=kind)

    return {"P": np.array([e.P for e in ests]), "L": np.array([e.L for e in ests]),
            "converged": np.array([e.converged for e in ests]), "N": pad(lambda e: e.N, np.int64),
            "mean": pad(lambda e: e.mean, np.float64), "var": pad(lambda e: e.var, np.float64)}


def run(s):
    c, kind = s["case"], s["kind"]
    if kind == "plain":
        return {"sums": np.array([mlmc.mlmc_level_sums_ex(l, c["M"], c["N"], 0, s["problem"], s["seed"],
                                                          precision=c["precision"])[0] for l in range(c["level"] + 1)])}
    if kind == "level":
        mlmc.mlmc_level_sums_async(c["level"], c["M"], c["N"], c["first"], s["problem"], s["seed"], s["sums"], s["ws"],
                                   s["bytes"], precision=c["precision"], d_y=s["y"],
                                   stream=torch.cuda.current_stream())
        return {"sums": s["sums"]} if s["y"] is None else {"sums": s["sums"], "y": s["y"]}
    if kind == "estimate":
        return _estimate_outputs([mlmc.mlmc_estimate(c["eps"], s["problem"], s["seed"], precision=c["precision"])])
    if kind == "batch":
        return _estimate_outputs(mlmc.mlmc_estimate_batch(s["problems"]))
    if kind == "cv":
        stream = torch.cuda.current_stream()
        mlmc.mlmc_cv_level_sums(s["cv"], c["level"], c["N"], 0, s["seed"], s["sums"], d_r=s["r"], stream=stream)
        mlmc.mlmc_cv_mean_sums(s["cv"], c["level"], c["replicates"], 0, s["seed"], s["mean"], stream=stream)
        return {"sums": s["sums"], "mean": s["mean"], "r": s["r"]}
    loss, grad = mlmc.mlmc_mlp_grad(s["params"], s["X"], s["Y"], c["rows"], stream=torch.cuda.current_stream())
    return {"loss": loss, "grad": grad}


# Operations of one fine step that no form of the method avoids: a normal (half of a Box--Muller
# pair: logarithm, root, sine and cosine, their products, a quarter of a Philox block's 20
# multiplies and 40 xors), its scaling, the step, the coarse sum, the payoff's functional, and a
# quarter of a coarse step.
FLOPS_STEP = 30.0
FLOPS_NETWORK = 2.0 * (16 * 64 + 64 * 64 + 64) + 128 * 8
# eps^2 times the fine steps of an adaptive estimate, by payoff (Euler--Maruyama, about)
ESTIMATE_STEPS = {"european": 1.6e3, "asian": 1.1e3, "lookback": 2.7e4, "digital": 1.0e2}


def work(case):
    kind = case["kind"]
    if kind == "plain":
        return {"bytes": 32.0 * (case["level"] + 1),
                "flops": FLOPS_STEP * case["N"] * sum(case["M"] ** l for l in range(case["level"] + 1))}
    if kind == "level":
        return {"bytes": 32.0 + (8.0 * case["N"] if case["per_sample"] else 0.0),
                "flops": FLOPS_STEP * case["N"] * case["M"] ** case["level"]}
    if kind == "estimate":
        return {"bytes": 400.0, "flops": FLOPS_STEP * ESTIMATE_STEPS[case["payoff"]] / case["eps"] ** 2}
    if kind == "batch":
        lo, hi = case["eps_lo"], case["eps_hi"]
        inv2 = (lo ** -2 - hi ** -2) / (2.0 * math.log(hi / lo))  # mean of eps^-2, eps log-uniform
        return {"bytes": 400.0 * case["n"],
                "flops": FLOPS_STEP * case["n"] * inv2 * sum(ESTIMATE_STEPS.values()) / 4.0}
    if kind == "cv":
        points = case["N"] + 65536.0 * case["replicates"]
        return {"bytes": 4.0 * case["N"], "flops": FLOPS_NETWORK * points + FLOPS_STEP * case["N"] * 4 ** case["level"]}
    return {"bytes": 68.0 * case["rows"] + 8.0 * 5313, "flops": 3.0 * FLOPS_NETWORK * case["rows"]}


# ------------------------------------------------------------------ the same outputs in 64 bits

_MASK = 0xFFFFFFFF


def _philox(c, key):
    """Philox4x32-10 on int64 tensors holding 32-bit words."""
    x, y, z, w = c
    k0, k1 = key & _MASK, (key >> 32) & _MASK
    for _ in range(10):
        a, b = x * 0xD2511F53, z * 0xCD9E8D57  # 64-bit products, wrapped; the shifts below mask the sign
        x, y, z, w = ((b >> 32) & _MASK) ^ y ^ k0, b & _MASK, ((a >> 32) & _MASK) ^ w ^ k1, a & _MASK
        k0, k1 = (k0 + 0x9E3779B9) & _MASK, (k1 + 0xBB67AE85) & _MASK
    return x, y, z, w


def _pair(xa, xb, stream32):
    if stream32:
        u1, u2 = (1.0 - (x & 0x7FFFFF).double() * 2.0 ** -23 for x in (xa, xb))
    else:
        u1, u2 = ((x.double() + 1.0) * 2.0 ** -32 for x in (xa, xb))
    rho = torch.sqrt(-2.0 * torch.log(u1))
    q = torch.round(4.0 * u2)  # 2 pi u2 = q pi/2 + t with |t| <= pi/4, the difference exact
    t = (2.0 * math.pi) * (u2 - 0.25 * q)
    ct, st, q = torch.cos(t), torch.sin(t), q.long() & 3
    c = torch.where(q == 0, ct, torch.where(q == 1, -st, torch.where(q == 2, -ct, st)))
    s = torch.where(q == 0, st, torch.where(q == 1, ct, torch.where(q == 2, -st, -ct)))
    return rho * c, rho * s


def _blocks(level, index, j, seed, stream32, tag=0):
    """The normals of Philox blocks j (tensor [J]) of counter indices index ([n]): [n, 4 J]."""
    i = index[:, None].expand(-1, len(j))
    zero = torch.zeros_like(i)
    x = _philox((zero + ((tag << 16) | level), zero + j[None, :], (i >> 32) & _MASK, i & _MASK), seed)
    z = _pair(x[0], x[1], stream32) + _pair(x[2], x[3], stream32)
    return torch.stack(z, dim=2).reshape(len(index), -1)


def _normals(level, M, first, n, j0, j1, seed, stream32):
    """Normals of fine steps 4 j0 .. 4 j1 of samples [first, first + n): [n, steps]."""
    nf, dev = M ** level, "cuda"
    s = torch.arange(first, first + n, device=dev)
    if nf >= 4:
        return _blocks(level, s, torch.arange(j0, j1, device=dev), seed, stream32)
    G = 4 // nf  # samples that share a block
    q0, q1 = first // G, (first + n - 1) // G + 1
    z = _blocks(level, torch.arange(q0, q1, device=dev), torch.zeros(1, dtype=torch.long, device=dev), seed, stream32)
    return z.reshape(-1, nf)[first - q0 * G:first - q0 * G + n]


class _Path:
    """A Euler--Maruyama or Milstein path's running functionals over consecutive pieces of steps."""

    def __init__(self, n, steps, scheme):
        self.S = torch.full((n,), S0, dtype=torch.float64, device="cuda")
        self.post, self.hi = torch.zeros_like(self.S), self.S.clone()
        self.h, self.n, self.scheme = T / steps, steps, scheme

    def take(self, z, root_h):
        """Steps with increments root_h z of the finest grid (already summed for the coarse path)."""
        dW = root_h * z
        d = R * self.h + SIGMA * dW
        if self.scheme == "milstein":
            d = d + 0.5 * SIGMA ** 2 * (dW * dW - self.h)
        v = self.S[:, None] * torch.cumprod(1.0 + d, dim=1)
        self.post += v.sum(dim=1)
        self.hi = torch.maximum(self.hi, v.amax(dim=1))
        self.S = v[:, -1].clone()

    def payoff(self, kind):
        disc = math.exp(-R * T)
        if kind == "digital":
            return disc * ((self.S > K).double() + 0.5 * (self.S == K).double())
        x = {"european": self.S, "lookback": self.hi,
             "asian": (self.post + 0.5 * (S0 - self.S)) / self.n}[kind]
        return disc * torch.clamp(x - K, min=0.0)


def _level_Y(case, level, first, n, seed):
    M, nf = case["M"], case["M"] ** level
    scheme, est = case.get("scheme", "em"), case.get("estimator", "coupled")
    fine, root_h = _Path(n, nf, scheme), math.sqrt(T / nf)
    anti = _Path(n, nf, scheme) if est == "antithetic" and level else None
    coarse = _Path(n, nf // M, scheme) if level and est != "single" else None
    piece = max(2, (1 << 22) // n // 2 * 2)  # Philox blocks at a time, whole coarse steps of M <= 8
    calls = max(1, nf // 4)
    for j in range(0, calls, piece):
        z = _normals(level, M, first, n, j, min(calls, j + piece), seed, case["precision"] != "fp64")
        fine.take(z, root_h)
        if anti:
            anti.take(z.reshape(n, -1, M).flip(2).reshape(n, -1), root_h)
        if coarse:
            coarse.take(z.reshape(n, -1, M).sum(dim=2), root_h)
    Y = fine.payoff(case["payoff"])
    if anti:
        Y = 0.5 * (Y + anti.payoff(case["payoff"]))
    return Y - coarse.payoff(case["payoff"]) if coarse else Y


def _level_exact(case, level, first, N, seed, keep=False):
    sums, ys = torch.zeros(4, dtype=torch.float64, device="cuda"), []
    chunk = max(1, min(N, (1 << 24) // case["M"] ** level, 1 << 22))
    for a in range(first, first + N, chunk):
        y = _level_Y(case, level, a, min(chunk, first + N - a), seed)
        sums += torch.stack([(y ** k).sum() for k in (1, 2, 3, 4)])
        if keep:
            ys.append(y)
    return (sums, torch.cat(ys)) if keep else (sums, None)


def _estimate_exact(case, seed):
    """The adaptive algorithm on exact level sums (M = 4, Lmin = 2, Lmax = 8, 10^4 samples first)."""
    M, eps, L, Lmax = 4, case["eps"], 2, 8
    case = dict(case, M=M)
    N, S, dN = [0] * 3, [np.zeros(4) for _ in range(3)], [10_000] * 3
    scale = (2.0 * M + 1.0) / (M + 1.0) if case["estimator"] == "antithetic" else 1.0

    def cost(l):
        return 1.0 if l == 0 else (M ** l + M ** (l - 1)) * scale

    def slope(y):
        x = np.arange(1, L + 1, dtype=np.float64)
        return ((x - x.mean()) * (y - y.mean())).sum() / ((x - x.mean()) ** 2).sum()

    while any(dN):
        for l, extra in enumerate(dN):
            if extra:
                S[l] = S[l] + _level_exact(case, l, N[l], extra, seed)[0].cpu().numpy()
                N[l] += extra
        n = np.array(N, dtype=np.float64)
        mean = np.array([s[0] for s in S]) / n
        var = np.maximum(np.array([s[1] for s in S]) / n - mean ** 2, 0.0)
        alpha = max(0.5, -slope(np.log(np.maximum(np.abs(mean[1:]), 1e-300)) / math.log(M)))
        beta = max(0.5, -slope(np.log(np.maximum(var[1:], 1e-300)) / math.log(M)))
        mf, vf, Ma, Mb = mean.copy(), list(var), M ** alpha, M ** beta
        for l in range(2, L + 1):
            mf[l] = max(abs(mf[l]), 0.5 * abs(mf[l - 1]) / Ma)
            vf[l] = max(vf[l], 0.5 * vf[l - 1] / Mb)

        def wanted():
            tot = sum(math.sqrt(v * cost(l)) for l, v in enumerate(vf))
            return [max(0, math.ceil(2.0 / eps ** 2 * math.sqrt(v / cost(l)) * tot) - (N[l] if l < len(N) else 0))
                    for l, v in enumerate(vf)]

        dN = wanted()
        bias = max(abs(mf[L]), abs(mf[L - 1]) / Ma) / (Ma - 1.0)
        if all(d <= 0.01 * k for d, k in zip(dN, N)) and bias > eps / math.sqrt(2.0) and L < Lmax:
            L += 1
            vf.append(vf[-1] / Mb)
            N.append(0)
            S.append(np.zeros(4))
            dN = wanted()
    top = mlmc.MLMC_MAX_LEVELS
    pad = np.zeros(top - L - 1)
    return {"P": np.array([mean.sum()]), "L": None, "converged": None, "N": None,
            "mean": np.concatenate([mean, pad])[None, :], "var": np.concatenate([var, pad])[None, :]}


def _net(theta, X):
    t = torch.as_tensor(theta, device=X.device).double()
    w1, b1, w2, b2, w3, b3 = torch.split(t, [1024, 64, 4096, 64, 64, 1])
    h = torch.nn.functional.gelu(X @ w1.reshape(64, 16).T + b1, approximate="tanh")
    h = torch.nn.functional.gelu(h @ w2.reshape(64, 64).T + b2, approximate="tanh")
    return h @ w3 + b3


def _levy(grid):
    """The Brownian-bridge coordinates of W at i T / 16, i = 0..16 (columns of grid)."""
    x, w = [grid[:, 16] / math.sqrt(T)], 16
    while w > 1:
        x += [(grid[:, a + w // 2] - 0.5 * (grid[:, a] + grid[:, a + w])) / math.sqrt(T * w / 64.0)
              for a in range(0, 16, w)]
        w //= 2
    return torch.stack(x, dim=1)


def _cv_exact(case, seed):
    level, nf = case["level"], 4 ** case["level"]
    theta = _network(seed)
    plain = dict(case, M=4, precision="fp32")
    sums, rs = torch.zeros(8, dtype=torch.float64, device="cuda"), []
    for a in range(0, case["N"], 1 << 18):
        n = min(1 << 18, case["N"] - a)
        Y = _level_Y(plain, level, a, n, seed)
        W = torch.cumsum(_normals(level, 4, a, n, 0, max(1, nf // 4), seed, True), dim=1) * math.sqrt(T / nf)
        grid = torch.zeros(n, 17, dtype=torch.float64, device="cuda")
        if nf >= 16:
            grid[:, 1:] = W[:, nf // 16 - 1::nf // 16]
        else:
            grid[:, 16 // nf::16 // nf] = W
            b0, count = max(1, nf // 4), (19 - nf) // 4
            zb = _blocks(level, torch.arange(a, a + n, device="cuda"),
                         torch.arange(b0, b0 + count, device="cuda"), seed, True)
            k, w = 0, 16 // nf
            while w > 1:
                for left in range(0, 16, w):
                    grid[:, left + w // 2] = (0.5 * (grid[:, left] + grid[:, left + w])
                                              + math.sqrt(T * w / 64.0) * zb[:, k])
                    k += 1
                w //= 2
        g = _net(theta, _levy(grid))
        r = Y - g
        sums += torch.stack([(r ** k).sum() for k in (1, 2, 3, 4)] + [Y.sum(), (Y * Y).sum(), g.sum(), (g * g).sum()])
        rs.append(r)
    z, k = [], 1
    for _ in range(16):
        z.append(k)
        k = k * 43833 % 65536
    i = torch.arange(65536, device="cuda")[:, None] * torch.tensor(z, device="cuda")[None, :] % 65536 * 65536
    mean = torch.zeros(2, dtype=torch.float64, device="cuda")
    for rep in range(case["replicates"]):
        # the lattice's shift: the words of blocks 0..3 of counter (j, rep, 0, tag 1 and level)
        j = torch.arange(4, device="cuda")
        D = torch.stack(_philox((j, j * 0 + rep, j * 0, j * 0 + ((1 << 16) | level)), seed), dim=1).reshape(-1)
        v = (i + D[None, :]) & _MASK
        v = torch.where(v < (1 << 31), 2 * v, 2 * (_MASK - v))
        q = _net(theta, torch.special.ndtri(((v >> 9).double() + 0.5) * 2.0 ** -23)).mean()
        mean += torch.stack([q, q * q])
    return {"sums": sums, "mean": mean, "r": torch.cat(rs)}


def exact(case, seed):
    kind = case["kind"]
    if kind == "plain":
        return {"sums": torch.stack([_level_exact(case, l, 0, case["N"], seed)[0] for l in range(case["level"] + 1)])}
    if kind == "level":
        sums, y = _level_exact(case, case["level"], case["first"], case["N"], seed, case["per_sample"])
        return {"sums": sums} if y is None else {"sums": sums, "y": y}
    if kind == "estimate":
        # FP32 sums move the sample counts themselves: only the FP64 estimates have a value here
        return _estimate_exact(case, seed) if case["precision"] == "fp64" else None
    if kind == "batch":
        return None
    if kind == "cv":
        return _cv_exact(case, seed)
    X, Y = _rows(case, seed)
    theta = torch.as_tensor(_network(seed), device="cuda").double().requires_grad_(True)
    loss = ((_net(theta, X.double()) - Y.double()) ** 2).mean()
    loss.backward()
    return {"loss": float(loss), "grad": theta.grad}
