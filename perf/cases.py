"""Performance cases: what users of the library run, through its public entry points.

A case is a dict with a "kind":

* "product"  one square product on a kept plan: both norm maps, plan, multiply
* "general"  one rectangular product C = alpha A B + beta C on a kept plan
* "chain"    X -> X^(2^steps) by squaring, each step planned from the norm map that the
             multiply before it wrote
* "batch"    many uneven instances on a kept batch (graph replay)
* "select"   the tau for a target error (learned prediction, error check, bisection),
             then the product at that tau
* "train"    Adam steps of the learned-tau network

Sizes, matrix families, leaf sizes and thresholds are those of bench.py, of the tests and of
the synthetic workloads (exponential and algebraic decay, near-sparse activations, the slowly
decaying Table 1 matrix, the VGG13 im2col shapes).  tau > 0 is absolute; ratio > 0 asks for the
tau at which that fraction of the block triples survives.
"""
import math

import numpy as np
import torch

import paper_2103_13042_gb300 as P

DEV = "cuda"


def listed():
    return [
        # the smallest single product: plain FP32, leaf 32; launches and latency count
        {"name": "product_fp32_n1024", "kind": "product", "n": 1024, "leaf": 32,
         "precision": "fp32", "family": "exp", "rate": 0.5, "tau": 1e-4, "ratio": 0.0,
         "schedule": "static"},
        # mixed precision on algebraic decay (bench.py --workload c2): an ordinary product
        {"name": "product_split_n8192", "kind": "product", "n": 8192, "leaf": 64,
         "precision": "bf16_split", "family": "alg", "rate": 3.0, "tau": 1e-2, "ratio": 0.0,
         "schedule": "static"},
        # the largest operands (bench.py default): bound by the bytes of A, B and C
        {"name": "product_fp16_n32768", "kind": "product", "n": 32768, "leaf": 128,
         "precision": "fp16", "family": "exp", "rate": 0.5, "tau": 1e-6, "ratio": 0.0,
         "schedule": "static"},
        # dense-ish skip set on near-sparse activations (bench.py --workload sparse): the
        # largest amount of tensor-core work
        {"name": "product_sparse_n16384", "kind": "product", "n": 16384, "leaf": 128,
         "precision": "bf16", "family": "sparse", "rate": 0.7, "tau": 0.0, "ratio": 0.5,
         "schedule": "groups"},
        # slow decay at a 10% valid ratio (bench.py --workload table2), FP16
        {"name": "product_slow_fp16_n8192", "kind": "product", "n": 8192, "leaf": 128,
         "precision": "fp16", "family": "slow", "rate": 0.1, "tau": 0.0, "ratio": 0.1,
         "schedule": "static"},
        # the same family in plain FP32: bound by the FP32 units
        {"name": "product_slow_fp32_n4096", "kind": "product", "n": 4096, "leaf": 64,
         "precision": "fp32", "family": "slow", "rate": 0.1, "tau": 0.0, "ratio": 0.3,
         "schedule": "static"},
        # a rectangular product: im2col of a convolution layer, near-sparse activations
        {"name": "general_bf16_conv", "kind": "general", "m": 256, "k": 1152, "n": 6400,
         "leaf": 64, "precision": "bf16", "family": "sparse", "rate": 0.05, "tau": 0.0,
         "ratio": 0.5, "alpha": 1.0, "beta": 0.0},
        # matrix powers at a ragged size, compensated TF32
        {"name": "chain_tf32x3_n3001", "kind": "chain", "n": 3001, "leaf": 64,
         "precision": "tf32x3", "rate": 0.2, "tau": 1e-6, "steps": 3},
        # serving: 256 uneven instances in one graph (bench.py --workload batch)
        {"name": "batch_split_256", "kind": "batch", "count": 256, "lo": 256, "hi": 4096,
         "leaf": 64, "precision": "bf16_split", "rel": 1e-6},
        # serving: few small instances; launches and latency count
        {"name": "batch_fp32_24_small", "kind": "batch", "count": 24, "lo": 64, "hi": 512,
         "leaf": 32, "precision": "fp32", "rel": 1e-6},
        # choosing tau for a target error, then the product
        {"name": "select_n4096", "kind": "select", "n": 4096, "leaf": 64, "family": "alg",
         "rate": 2.5, "target": 1e-5},
        # training the learned-tau network: minibatches of 256
        {"name": "train_b256", "kind": "train", "samples": 20000, "batch": 256, "steps": 64,
         "lr": 1e-3, "quantile": 0.1},
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["product"] * 6 + ["general"] * 2 + ["chain", "batch", "batch", "select",
                                                           "train"])
    if kind == "product":
        family = rng.choice(["exp", "exp", "alg", "alg", "sparse", "slow"])
        precision = rng.choice(sorted(P.PRECISIONS))
        leaf = rng.choice([32, 64, 128] if precision == "fp32" else [64, 128])
        case = {"kind": kind, "leaf": leaf, "precision": precision, "family": family,
                "tau": 0.0, "ratio": 0.0, "schedule": rng.choice(["static", "static", "dynamic",
                                                                  "groups"])}
        if family == "exp":
            case.update(n=_logint(rng, 256, 32768), rate=round(rng.uniform(0.1, 1.5), 3),
                        tau=10.0 ** rng.uniform(-7, -2))
        elif family == "alg":
            case.update(n=_logint(rng, 256, 12288), rate=round(rng.uniform(2.0, 4.0), 3),
                        tau=10.0 ** rng.uniform(-6, -1))
        elif family == "sparse":
            top = 4096 if precision in ("fp32", "tf32x3") else 16384
            case.update(n=_logint(rng, 512, top), rate=0.7, ratio=round(rng.uniform(0.1, 0.5), 3))
        else:
            top = 4096 if precision in ("fp32", "tf32x3") else 8192
            case.update(n=_logint(rng, 512, top), rate=0.1,
                        ratio=round(rng.uniform(0.05, 0.3), 3))
        if case["n"] / case["leaf"] > 1024:
            case["leaf"] = 64
        return case
    if kind == "general":
        precision = rng.choice(sorted(P.PRECISIONS))
        beta = rng.choice([0.0, 0.0, 0.5])
        family, k, n = rng.choice(["sparse", "exp"]), _logint(rng, 300, 4608), \
            _logint(rng, 200, 25600)
        return {"kind": kind, "m": _logint(rng, 100, 1024), "k": k, "n": n,
                "leaf": rng.choice([32, 64, 128] if precision == "fp32" else [64, 128]),
                "precision": precision, "family": family,
                "rate": rng.uniform(5.0, 40.0) / (k if family == "sparse" else max(k, n)),
                "tau": 0.0,
                "ratio": round(rng.uniform(0.1, 0.5), 3),
                "alpha": rng.choice([1.0, -1.5]) if beta else 1.0, "beta": beta}
    if kind == "chain":
        precision = rng.choice(["fp32", "tf32x3", "bf16_split"])
        return {"kind": kind, "n": _logint(rng, 500, 5000), "leaf": rng.choice([64, 128]),
                "precision": precision, "rate": round(rng.uniform(0.1, 0.5), 3),
                "tau": 10.0 ** rng.uniform(-7, -5), "steps": rng.choice([2, 3])}
    if kind == "batch":
        precision = rng.choice(["fp32", "bf16", "fp16", "bf16_split", "bf16_split"])
        lo = _logint(rng, 48, 256)
        return {"kind": kind, "count": _logint(rng, 8, 128), "lo": lo,
                "hi": lo * rng.choice([4, 8, 12]),
                "leaf": rng.choice([32, 64] if precision == "fp32" else [64, 128]),
                "precision": precision, "rel": 10.0 ** rng.uniform(-7, -5)}
    if kind == "select":
        family = rng.choice(["exp", "alg"])
        return {"kind": kind, "n": _logint(rng, 1024, 8192), "leaf": 64, "family": family,
                "rate": round(rng.uniform(0.2, 1.5) if family == "exp" else rng.uniform(2.0, 4.0),
                              3),
                "target": 10.0 ** rng.uniform(-6, -3)}
    return {"kind": "train", "samples": _logint(rng, 2000, 20000),
            "batch": rng.choice([64, 100, 128, 256]), "steps": _logint(rng, 8, 78),
            "lr": rng.choice([1e-3, 2e-4]), "quantile": 0.1}


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _matrix(rows, cols, family, rate, g, stretch=1.0):
    """One operand of a family, drawn in row chunks (bounded temporaries)."""
    out = torch.empty(rows, cols, device=DEV, dtype=torch.float32)
    j = torch.arange(cols, device=DEV, dtype=torch.float32)
    step = max(1, (1 << 26) // cols)
    for r0 in range(0, rows, step):
        r1 = min(rows, r0 + step)
        shape = (r1 - r0, cols)
        if family == "sparse":      # ReLU(N(0, 1)), a share `rate` of the rest zeroed
            z = torch.randn(shape, generator=g, device=DEV).clamp_min_(0.0)
            z *= torch.rand(shape, generator=g, device=DEV) >= rate
            out[r0:r1] = z
            continue
        i = torch.arange(r0, r1, device=DEV, dtype=torch.float32) * stretch
        d = (i[:, None] - j[None, :]).abs()
        if family == "exp":         # exp(-rate d) N(0, 1)
            out[r0:r1] = torch.exp(-rate * d) * torch.randn(shape, generator=g, device=DEV)
        else:
            sign = torch.randint(0, 2, shape, generator=g, device=DEV) * 2.0 - 1.0
            if family == "alg":     # (d + 1)^-rate, random signs
                out[r0:r1] = (d + 1.0).pow(-rate) * sign
            else:                   # 0.1 / (d^rate + 1), random signs and sizes
                u = torch.rand(shape, generator=g, device=DEV) * 0.5 + 0.5
                out[r0:r1] = 0.1 / (d.pow(rate) + 1.0) * sign * u
    return out


def _norms64(X, leaf):
    """Block norms in FP64, in row chunks of whole blocks."""
    rows, cols = X.shape
    bc = -(-cols // leaf)
    out = []
    step = leaf * max(1, (1 << 25) // (leaf * bc * leaf))
    for r0 in range(0, rows, step):
        x = X[r0:r0 + step].double()
        br = -(-x.shape[0] // leaf)
        x = torch.nn.functional.pad(x, (0, bc * leaf - cols, 0, br * leaf - x.shape[0]))
        out.append(x.square_().view(br, leaf, bc, leaf).sum((1, 3)).sqrt_())
    return torch.cat(out)


def _tau(case, A, B):
    """The case's threshold: absolute, or midway between two neighbouring norm products at the
    wanted valid ratio."""
    if case["ratio"] == 0.0:
        return case["tau"]
    nA, nB = _norms64(A, case["leaf"]), _norms64(B, case["leaf"])
    p = (nA[:, :, None] * nB[None, :, :]).reshape(-1).sort().values
    at = min(p.numel() - 1, max(1, int(round(p.numel() * (1.0 - case["ratio"])))))
    return 0.5 * (p[at - 1].item() + p[at].item())


def _operands(case, seed):
    kind = case["kind"]
    if kind == "product":
        n, f, r = case["n"], case["family"], case["rate"]
        return _matrix(n, n, f, r, _gen(2 * seed)), _matrix(n, n, f, r, _gen(2 * seed + 1))
    if kind == "general":           # weights smooth in the channel index, then activations
        m, k, n = case["m"], case["k"], case["n"]
        A = _matrix(m, k, "exp", case["rate"], _gen(2 * seed), k / m)
        if case["family"] == "sparse":
            return A, _matrix(k, n, "sparse", 0.7, _gen(2 * seed + 1))
        return A, _matrix(k, n, "exp", case["rate"], _gen(2 * seed + 1), n / k)
    if kind == "chain":
        return 0.5 * _matrix(case["n"], case["n"], "exp", case["rate"], _gen(seed))
    n, f, r = case["n"], case["family"], case["rate"]      # select
    return _matrix(n, n, f, r, _gen(2 * seed)), _matrix(n, n, f, r, _gen(2 * seed + 1))


def _start_c(case, seed):
    """The C that a beta != 0 product adds to."""
    return torch.randn(case["m"], case["n"], generator=_gen(7 * seed + 3), device=DEV)


def _instances(case, seed):
    """Batch: the instances' sizes, operands and thresholds.  Sizes depend on the case alone."""
    r = np.random.RandomState(case["count"] * 7919 + case["lo"])
    ns, As, Bs, taus = [], [], [], []
    for t in range(case["count"]):
        n = int(round(math.exp(r.uniform(math.log(case["lo"]), math.log(case["hi"])))))
        family = "exp" if r.uniform() < 0.5 else "alg"
        rate = r.uniform(0.2, 1.5) if family == "exp" else r.uniform(2.0, 4.0)
        g = _gen(seed * 1000 + t)
        ns.append(n)
        As.append(_matrix(n, n, family, rate, g))
        Bs.append(_matrix(n, n, family, rate, g))
    scale = torch.stack([torch.linalg.vector_norm(a) * torch.linalg.vector_norm(b)
                         for a, b in zip(As, Bs)]).double().tolist()
    for n, s in zip(ns, scale):
        taus.append(case["rel"] * s / -(-n // case["leaf"]))
    return ns, As, Bs, taus


def _arena_layout(ns):
    """Offsets (floats, 256-byte aligned) of the instances' outputs in one buffer."""
    offs, total = [], 0
    for n in ns:
        offs.append(total)
        total += -(-n * n // 64) * 64
    return offs, total


def _train_data(case, seed):
    """Histogram features with a target error, and a tau that follows them with noise."""
    g = _gen(seed)
    n = case["samples"]
    bins = torch.arange(64, device=DEV, dtype=torch.float32)
    c = torch.rand(n, 1, generator=g, device=DEV) * 40 + 8
    w = torch.rand(n, 1, generator=g, device=DEV) * 8 + 2
    h = torch.exp(-((bins - c) / w) ** 2) + 0.002 * torch.rand(n, 64, generator=g, device=DEV)
    h = h / h.sum(1, keepdim=True)
    e = -1.0 - 6.0 * torch.rand(n, 1, generator=g, device=DEV)
    X = torch.cat([h, e], 1).contiguous()
    Y = (e[:, 0] - 0.05 * c[:, 0] + 0.3 * torch.randn(n, generator=g, device=DEV)).contiguous()
    sizes = (65, 64, 64, 1)
    parts = []
    for a, b in zip(sizes[:-1], sizes[1:]):
        for count in (a * b, b):
            parts.append((torch.rand(count, generator=g, device=DEV) * 2 - 1) / math.sqrt(a))
    W = torch.cat(parts).contiguous()
    need = case["steps"] * case["batch"]
    perms = [torch.randperm(n, generator=g, device=DEV) for _ in range(-(-need // n))]
    return X, Y, W, torch.cat(perms)[:need].to(torch.int32).contiguous()


def prepare(case, seed):
    kind, seed = case["kind"], int(seed)
    s = {"kind": kind, "case": case}
    if kind == "product":
        n, leaf = case["n"], case["leaf"]
        A, B = _operands(case, seed)
        plan = P.Plan(n, leaf, P.PRECISIONS[case["precision"]])
        plan.set_schedule(case["schedule"])
        bd = -(-n // leaf)
        s.update(A=A, B=B, tau=_tau(case, A, B), plan=plan, C=torch.empty_like(A),
                 nA=torch.empty(bd, bd, device=DEV, dtype=torch.float64),
                 nB=torch.empty(bd, bd, device=DEV, dtype=torch.float64))
    elif kind == "general":
        A, B = _operands(case, seed)
        m, k, n, leaf = case["m"], case["k"], case["n"], case["leaf"]
        s.update(A=A, B=B, tau=_tau(case, A, B), C=_start_c(case, seed),
                 plan=P.GeneralPlan(m, k, n, leaf, P.PRECISIONS[case["precision"]]))
        s.update(nA=P.spamm_normmap_rect(A, leaf), nB=P.spamm_normmap_rect(B, leaf))
    elif kind == "chain":
        n, leaf = case["n"], case["leaf"]
        X = _operands(case, seed)
        bd = -(-n // leaf)
        s.update(X=X, nX=torch.empty(bd, bd, device=DEV, dtype=torch.float64),
                 plan=P.GeneralPlan(n, n, n, leaf, P.PRECISIONS[case["precision"]]),
                 Y=[torch.empty_like(X) for _ in range(case["steps"])],
                 nY=[torch.empty(bd, bd, device=DEV, dtype=torch.float64)
                     for _ in range(case["steps"])])
    elif kind == "batch":
        ns, As, Bs, taus = _instances(case, seed)
        offs, total = _arena_layout(ns)
        arena = torch.zeros(total, device=DEV, dtype=torch.float32)
        Cs = [arena[o:o + n * n].view(n, n) for o, n in zip(offs, ns)]
        s.update(As=As, Bs=Bs, Cs=Cs, arena=arena, taus=taus,
                 batch=P.Batch(ns, case["leaf"], P.PRECISIONS[case["precision"]], graph=True))
    elif kind == "select":
        A, B = _operands(case, seed)
        s.update(A=A, B=B, plan=P.Plan(case["n"], case["leaf"], P.FP32),
                 nA=P.spamm_normmap(A, case["leaf"]), nB=P.spamm_normmap(B, case["leaf"]),
                 W=P.load_tau_weights(), scratch=torch.empty_like(A), C=torch.empty_like(A))
    else:
        X, Y, W, idx = _train_data(case, seed)
        s.update(X=X, Y=Y, W=W, idx=idx, m=torch.zeros_like(W), v=torch.zeros_like(W), t=0)
    return s


def run(s):
    case, kind = s["case"], s["kind"]
    if kind == "product":
        P.spamm_normmap_pair(s["A"], s["B"], case["leaf"], s["nA"], s["nB"])
        s["plan"].plan_multiply(s["nA"], s["nB"], s["tau"], s["A"], s["B"], s["C"])
        return {"C": s["C"], "nA": s["nA"], "nB": s["nB"]}
    if kind == "general":
        P.spamm_normmap_rect(s["A"], case["leaf"], s["nA"])
        P.spamm_normmap_rect(s["B"], case["leaf"], s["nB"])
        s["plan"].plan_multiply(s["nA"], s["nB"], s["tau"], s["A"], s["B"], s["C"],
                                alpha=case["alpha"], beta=case["beta"])
        return {"C": s["C"], "nA": s["nA"], "nB": s["nB"]}
    if kind == "chain":
        P.spamm_normmap(s["X"], case["leaf"], s["nX"])
        X, nX = s["X"], s["nX"]
        for Y, nY in zip(s["Y"], s["nY"]):
            s["plan"].plan_multiply(nX, nX, case["tau"], X, X, Y, normC=nY)
            X, nX = Y, nY
        return {"powers": s["Y"], "nX": s["nX"]}
    if kind == "batch":
        s["batch"].run(s["As"], s["Bs"], s["Cs"], s["taus"])
        return {"C": s["arena"]}
    if kind == "select":
        tau, evals, err = s["plan"].tau_select(s["nA"], s["nB"], s["A"], s["B"], case["target"],
                                               s["W"], s["scratch"])
        s["plan"].plan_multiply(s["nA"], s["nB"], tau, s["A"], s["B"], s["C"])
        return {"C": s["C"], "tau": tau, "evals": evals, "err": err}
    hist = P.spamm_mlp_train(s["W"], s["m"], s["v"], s["t"], s["X"], s["Y"], s["idx"],
                             case["steps"], case["batch"], case["lr"], case["quantile"])
    s["t"] += case["steps"]
    return {"loss": hist, "W": s["W"], "m": s["m"], "v": s["v"]}


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------

def _decay_norm(db, leaf, family, rate):
    """Expected norm of a block `db` block diagonals from the diagonal."""
    off = np.arange(-leaf + 1, leaf, dtype=np.float64)
    count = leaf - np.abs(off)
    d = np.abs(db * leaf + off)
    mag = np.exp(-rate * d) if family == "exp" else (d + 1.0) ** -rate
    return math.sqrt(float((mag * mag * count).sum()))


def _decay_survivors(n, leaf, family, rate, tau):
    """Triples with p >= tau for the expected norms of a decay pair (Toeplitz in the blocks)."""
    bd = -(-n // leaf)
    v = np.array([_decay_norm(d, leaf, family, rate) for d in range(bd)])
    if tau <= 0.0:
        return bd ** 3
    # v falls with d: for a block at distance d, its partners are those within reach[d]
    reach = np.array([int(np.searchsorted(-v, -tau / max(x, 1e-300), side="right")) - 1
                      for x in v])
    k = np.arange(bd)
    total = 0
    for d in range(bd):
        if reach[d] < 0:
            break
        cols = np.minimum(bd - 1, k + reach[d]) - np.maximum(0, k - reach[d]) + 1
        rows = (k + d < bd).astype(np.int64) + ((k - d >= 0) & (d > 0))
        total += int((rows * cols).sum())
    return total


def work(case):
    kind = case["kind"]
    if kind == "product":
        n, leaf = case["n"], case["leaf"]
        if case["ratio"] > 0.0:
            flops = case["ratio"] * 2.0 * n ** 3
        else:
            flops = 2.0 * min(leaf, n) ** 3 * _decay_survivors(n, leaf, case["family"],
                                                               case["rate"], case["tau"])
        return {"bytes": 12.0 * n * n + 16.0 * (-(-n // leaf)) ** 2, "flops": flops}
    if kind == "general":
        m, k, n = case["m"], case["k"], case["n"]
        c = 8.0 if case["beta"] else 4.0
        return {"bytes": 4.0 * (m * k + k * n) + c * m * n,
                "flops": case["ratio"] * 2.0 * m * k * n}
    if kind == "chain":
        n, leaf, s = case["n"], case["leaf"], case["steps"]
        tri = _decay_survivors(n, leaf, "exp", case["rate"], 4.0 * case["tau"])
        return {"bytes": 4.0 * n * n * (1 + s), "flops": 2.0 * leaf ** 3 * tri * s}
    if kind == "batch":
        r = np.random.RandomState(case["count"] * 7919 + case["lo"])
        total, flops = 0.0, 0.0
        for _ in range(case["count"]):
            n = int(round(math.exp(r.uniform(math.log(case["lo"]), math.log(case["hi"])))))
            family = "exp" if r.uniform() < 0.5 else "alg"
            rate = r.uniform(0.2, 1.5) if family == "exp" else r.uniform(2.0, 4.0)
            total += 12.0 * n * n
            bd = -(-n // case["leaf"])
            ab = bd * _decay_norm(0, case["leaf"], family, rate) ** 2
            flops += 2.0 * case["leaf"] ** 3 * _decay_survivors(n, case["leaf"], family, rate,
                                                                case["rel"] * ab / bd)
        return {"bytes": total, "flops": flops}
    if kind == "select":
        n, leaf = case["n"], case["leaf"]
        tri = _decay_survivors(n, leaf, case["family"], case["rate"], case["target"])
        return {"bytes": 12.0 * n * n, "flops": 2.0 * leaf ** 3 * tri}
    samples = case["steps"] * case["batch"]
    return {"bytes": 4.0 * (66.0 * samples + 6 * 8449.0), "flops": 6.0 * 8384.0 * samples}


# ---------------------------------------------------------------------------
# The same results in 64 bits
# ---------------------------------------------------------------------------

def _product64(A, B, nA, nB, leaf, keep):
    """sum_k A[I,k] B[k,J] over the block triples that keep(k) -> [bm, bn] selects."""
    m, n = A.shape[0], B.shape[1]
    bm, bk, bn = nA.shape[0], nA.shape[1], nB.shape[1]
    C = torch.zeros(m, n, device=DEV, dtype=torch.float64)
    ri = torch.arange(m, device=DEV) // leaf
    ci = torch.arange(n, device=DEV) // leaf
    for k in range(bk):
        M = keep(nA[:, k, None] * nB[None, k, :])
        rows, cols = M.any(1), M.any(0)
        if not bool(rows.any()):
            continue
        ks = slice(k * leaf, (k + 1) * leaf)
        if bool(rows.all()) and bool(cols.all()):
            T = torch.mm(A[:, ks].double(), B[ks].double())
            if not bool(M.all()):
                T *= M.repeat_interleave(leaf, 0)[:m].repeat_interleave(leaf, 1)[:, :n]
            C += T
            continue
        r, c = rows[ri].nonzero()[:, 0], cols[ci].nonzero()[:, 0]
        T = torch.mm(A[r][:, ks].double(), B[ks][:, c].double())
        T *= M[ri[r]][:, ci[c]]
        C[r[:, None], c[None, :]] += T
    return C


def _select64(case, seed):
    """Certified tau, the network's prediction, its error check and the bisection, in FP64."""
    A, B = _operands(case, seed)
    leaf, eps = case["leaf"], case["target"]
    nA, nB = _norms64(A, leaf), _norms64(B, leaf)
    bd = nA.shape[0]
    ab = float(nA.square().sum().sqrt() * nB.square().sum().sqrt())
    p = nA[:, :, None] * nB[None, :, :]                # [i, k, j]

    def bound2(t):
        return float((p * (p < t)).sum(1).square_().sum().sqrt())

    lo, hi = -60.0, 0.0
    for _ in range(36):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if bound2(ab * 10.0 ** mid) <= 1e-11 * ab else (lo, mid)
    ref = ab * 10.0 ** lo
    evals = 0

    def err(t):
        nonlocal evals
        evals += 1
        if t <= ref:
            return 0.0
        band = _product64(A, B, nA, nB, leaf, lambda q: (q >= ref) & (q < t))
        return float(torch.linalg.vector_norm(band)) / ab

    bins = (-torch.log2((p * (1.0 / ab)).clamp_min(1e-300))).floor().clamp_(0, 63).long()
    x = torch.cat([torch.bincount(bins.reshape(-1), minlength=64).double() / bd ** 3,
                   torch.tensor([math.log10(eps)], device=DEV, dtype=torch.float64)])
    del bins
    y = float(_forward64(P.load_tau_weights().double(), x[None])[0])
    t = 10.0 ** y * ab
    e = err(t)
    if e > eps:
        first, lo, hi, lo_err = evals, 0.0, eps * ab, 0.0
        e = err(hi)
        if e <= eps:
            while e <= eps and evals - first < 40:
                lo, lo_err, hi = hi, e, hi * 10.0
                e = err(hi)
        else:
            t = hi / 10.0
            while evals - first < 40 and t > 0.0:
                e = err(t)
                if e <= eps:
                    lo, lo_err = t, e
                    break
                hi, t = t, t / 10.0
        while lo > 0.0 and hi / lo > 1.01 and evals - first < 40:
            mid = math.sqrt(lo * hi)
            e = err(mid)
            if e <= eps:
                lo, lo_err = mid, e
            else:
                hi = mid
        t, e = lo, lo_err
    C = _product64(A, B, nA, nB, leaf, lambda q: ~(q < t))
    return {"C": C, "tau": t, "evals": None, "err": e}


def _forward64(W, x):
    at, h = 0, x
    for a, b in ((65, 64), (64, 64), (64, 1)):
        w, bias = W[at:at + a * b].view(b, a), W[at + a * b:at + a * b + b]
        at += a * b + b
        h = h @ w.T + bias
        if b > 1:
            h = torch.nn.functional.gelu(h)
    return h[:, 0]


def _train64(case, seed):
    X, Y, W, idx = _train_data(case, seed)
    X, Y, W, q = X.double(), Y.double(), W.double(), case["quantile"]
    m, v, losses = torch.zeros_like(W), torch.zeros_like(W), []
    for t in range(case["steps"]):
        at = idx[t * case["batch"]:(t + 1) * case["batch"]].long()
        W.requires_grad_(True)
        r = Y[at] - _forward64(W, X[at])
        loss = torch.where(r > 0, q * r, (q - 1.0) * r).mean()
        g, = torch.autograd.grad(loss, W)
        W = W.detach()
        m = 0.9 * m + 0.1 * g
        v = 0.999 * v + 0.001 * g * g
        W = W - case["lr"] * (m / (1 - 0.9 ** (t + 1))) / ((v / (1 - 0.999 ** (t + 1))).sqrt() + 1e-8)
        losses.append(loss.detach())
    return {"loss": torch.stack(losses), "W": W, "m": m, "v": v}


def exact(case, seed):
    kind, seed = case["kind"], int(seed)
    if kind == "train":
        return _train64(case, seed)
    if kind == "select":
        return _select64(case, seed)
    if kind == "chain":
        X, leaf = _operands(case, seed), case["leaf"]
        nX = _norms64(X, leaf)
        powers, X, n = [], X.double(), nX
        for _ in range(case["steps"]):
            X = _product64(X, X, n, n, leaf, lambda q: ~(q < case["tau"]))
            n = _norms64(X, leaf)
            powers.append(X)
        return {"powers": powers, "nX": nX}
    if kind == "batch":
        ns, As, Bs, taus = _instances(case, seed)
        offs, total = _arena_layout(ns)
        arena = torch.zeros(total, device=DEV, dtype=torch.float64)
        for o, n, A, B, tau in zip(offs, ns, As, Bs, taus):
            nA, nB = _norms64(A, case["leaf"]), _norms64(B, case["leaf"])
            arena[o:o + n * n] = _product64(A, B, nA, nB, case["leaf"],
                                            lambda q: ~(q < tau)).reshape(-1)
        return {"C": arena}
    A, B = _operands(case, seed)
    leaf, tau = case["leaf"], _tau(case, A, B)
    nA, nB = _norms64(A, leaf), _norms64(B, leaf)
    C = _product64(A, B, nA, nB, leaf, lambda q: ~(q < tau))
    if kind == "general":
        C = case["alpha"] * C
        if case["beta"]:
            C += case["beta"] * _start_c(case, seed).double()
    return {"C": C, "nA": nA, "nB": nB}
