"""The work that a user of this library has it do, as a list of cases: bulk and
small encodes in every projection precision, encodes of host buffers, a burst
of serving requests, distance estimates from codes, the multi-stage bounds and
the fit.  Inputs follow the seeded recipe of the synthetic workloads (a
power-law spectrum under a Haar rotation, here with a non-zero mean).
"""
import math

import numpy as np
import torch

import paper_2509_12086_gb300 as P

F64 = torch.float64


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # one vector arriving at a resident collection: launches and latency
        dict(name="encode_1", kind="encode", n=1, d=960, alpha=0.8, bits=4.0, rounds=6,
             precision="fp32"),
        # the small collection of the test configurations, whole
        dict(name="encode_10k_d128", kind="encode", n=10_000, d=128, alpha=1.0, bits=4.0, rounds=6,
             precision="fp32"),
        # the benchmark's bulk encode
        dict(name="encode_1m_d960", kind="encode", n=1_000_000, d=960, alpha=0.8, bits=4.0,
             rounds=6, precision="fp32"),
        # an insert batch of a wide collection, BF16 projection, ragged row count
        dict(name="encode_100k_d1536_bf16", kind="encode", n=100_003, d=1536, alpha=0.6, bits=2.0,
             rounds=6, precision="bf16"),
        # the widest configuration at one bit per dimension, FP8 projection
        dict(name="encode_65k_d3072_fp8", kind="encode", n=65_537, d=3072, alpha=0.5, bits=1.0,
             rounds=6, precision="fp8"),
        # the same rows at eight bits: one long segment
        dict(name="encode_20k_d3072_8b", kind="encode", n=20_011, d=3072, alpha=0.5, bits=8.0,
             rounds=6, precision="fp32"),
        # rows and outputs in page-locked host memory
        dict(name="encode_host_100k_d960", kind="encode_host", n=100_000, d=960, alpha=0.8,
             bits=4.0, rounds=6, precision="fp32"),
        # a burst of insert requests over three resident collections
        dict(name="serve_48_requests", kind="serve", requests=48, most=8192, alpha=0.8,
             precision="bf16"),
        # one query against a collection
        dict(name="estimate_1q_1m", kind="estimate", nq=1, n=1_000_000, d=960, alpha=0.8, bits=4.0,
             prefix=0),
        # the benchmark's estimator batch
        dict(name="estimate_100q_100k", kind="estimate", nq=100, n=100_000, d=960, alpha=0.8,
             bits=4.0, prefix=0),
        # the multi-stage bounds a search prunes with
        dict(name="staged_10q_100k", kind="staged", nq=10, n=100_000, d=960, alpha=0.8, bits=4.0,
             m_conf=2.0),
        # the fit of a collection's model
        dict(name="fit_50k_d960", kind="fit", n=50_000, d=960, alpha=0.8, bits=4.0),
    ]


def _log_int(rng, lo, hi):
    return int(min(hi, max(lo, round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _dim(rng, lo=64, hi=3072, step=4):
    return max(lo, _log_int(rng, lo, hi) // step * step)


def draw(rng):
    kind = rng.choices(["encode", "encode_host", "serve", "estimate", "staged", "fit"],
                       [10, 2, 2, 5, 2, 2])[0]
    alpha = round(rng.uniform(0.5, 1.0), 2)
    bits = rng.choice([1.0, 2.0, 2.5, 3.0, 4.0, 4.0, 6.0, 8.0])
    if kind in ("encode", "encode_host"):
        precision = rng.choice(["fp32", "fp32", "fp32", "bf16", "bf16", "fp8", "fp32_simt"])
        # the tensor-core forms take d % 4 == 0, the CUDA-core form any d
        d = _dim(rng, step=1 if precision == "fp32_simt" else 4)
        most = min(1_000_000, 3 * 10 ** 11 // (d * d), 3 * 10 ** 8 // d)
        if precision == "fp32_simt":
            most = min(most, 5 * 10 ** 10 // (d * d))
        if kind == "encode_host":
            most = min(most, 10 ** 8 // d)
        return dict(kind=kind, n=_log_int(rng, 1, max(1, most)), d=d, alpha=alpha, bits=bits,
                    rounds=rng.choice([6, 6, 6, 1, 3, 10]), precision=precision)
    if kind == "serve":
        return dict(kind=kind, requests=rng.randint(4, 64), most=_log_int(rng, 64, 8192),
                    alpha=alpha, precision=rng.choice(["bf16", "fp32"]))
    if kind == "fit":
        d = _dim(rng, hi=960)
        return dict(kind=kind, n=_log_int(rng, 4 * d, 50_000), d=d, alpha=alpha, bits=bits)
    d = _dim(rng, hi=1536)
    nq = _log_int(rng, 1, 1000)
    n = _log_int(rng, 1000, min(1_000_000, 9 * 10 ** 9 // (d * nq)))
    if kind == "estimate":
        return dict(kind=kind, nq=nq, n=n, d=d, alpha=alpha, bits=bits,
                    prefix=rng.choice([0, 0, 0, 1, 2, 4]))
    return dict(kind=kind, nq=min(nq, 100), n=min(n, 100_000), d=d, alpha=alpha, bits=bits,
                m_conf=rng.choice([0.5, 2.0, 3.0]))


# ---------------------------------------------------------------- the inputs
def _gen(seed, salt, device="cuda"):
    return torch.Generator(device=device).manual_seed((int(seed) * 1_000_003 + salt) % (1 << 62))


def _haar(n, g):
    """A Haar orthogonal n x n matrix in 64 bits."""
    q, r = torch.linalg.qr(torch.randn(n, n, generator=g, dtype=F64, device="cuda"))
    s = torch.sign(torch.diagonal(r))
    s[s == 0] = 1.0
    return q * s


class _Data:
    """A distribution of rows: x = c + z diag(sqrt(lambda)) Q^T."""

    def __init__(self, d, alpha, seed, salt=0):
        self.d, self.seed, self.salt = d, seed, salt
        self.lam = torch.arange(1, d + 1, dtype=F64, device="cuda").pow(-alpha)
        self.Q = _haar(d, _gen(seed, salt + 1))
        self.c = 0.1 * torch.randn(d, generator=_gen(seed, salt + 2), dtype=F64, device="cuda")

    def rows(self, n, salt):
        M = (self.lam.sqrt()[:, None] * self.Q.T).float()
        c = self.c.float()
        X = torch.empty(n, self.d, device="cuda")
        step = 1 << 17
        tf32 = torch.backends.cuda.matmul.allow_tf32
        torch.backends.cuda.matmul.allow_tf32 = False
        try:
            for i in range(0, n, step):
                m = min(step, n - i)
                z = torch.randn(m, self.d, generator=_gen(self.seed, self.salt + salt + 1000 * (1 + i // step)),
                                device="cuda")
                X[i:i + m] = z @ M + c
        finally:
            torch.backends.cuda.matmul.allow_tf32 = tf32
        return X


class _Kept:
    """What 64-bit checks need of a model: mean, W, basis and the kept segments."""


def _model(data, bits, rounds=6, precision="fp32"):
    """The model of a distribution whose mean, principal directions and
    variances are known, as a fit on plenty of rows would return it."""
    d = data.d
    plan, _ = P.saq_plan_search(data.lam.cpu().numpy(), int(round(bits * d)))
    W, basis = [], []
    for k, (start, length, b) in enumerate(plan):
        if b > 0:
            V = data.Q[:, start:start + length].T
            W.append(_haar(length, _gen(data.seed, data.salt + 10 + k)) @ V)
            basis.append(V)
    W = torch.cat(W) if W else torch.zeros(0, d, dtype=F64, device="cuda")
    basis = torch.cat(basis) if basis else W
    m = P.saq_model_create(d, data.c.cpu().numpy(), W.cpu().numpy(), plan, data.lam.cpu().numpy(),
                           rounds=rounds, precision=precision,
                           basis=basis.cpu().numpy() if len(basis) else None)
    kept = _Kept()
    kept.mean, kept.W, kept.basis, kept.rounds = data.c, W, basis, rounds
    kept.segs = [(s, l, b) for s, l, b in plan if b > 0]
    kept.sigma = torch.cat([data.lam[s:s + l] for s, l, _ in kept.segs]).sqrt() if kept.segs else None
    return m, kept


# the serving run's collections: dimensions and bits
_COLLECTIONS = ((128, 4.0), (960, 4.0), (1536, 2.0))


def _serve_sizes(case):
    """(collection, rows) of every request: log-uniform sizes, the same for every seed."""
    g = np.random.default_rng([case["requests"], case["most"]])
    sizes = np.exp(g.uniform(0.0, math.log(case["most"]), case["requests"])).astype(int)
    return [(int(g.integers(0, 3)) if i >= 3 else i, max(1, int(n))) for i, n in enumerate(sizes)]


def prepare(case, seed):
    kind = case["kind"]
    st = {"kind": kind, "case": case}
    if kind == "serve":
        reqs = _serve_sizes(case)
        st["models"], st["kept"], st["X"], st["out"] = [], [], [], []
        for c, (d, bits) in enumerate(_COLLECTIONS):
            data = _Data(d, case["alpha"], seed, 100_000 * (c + 1))
            m, kept = _model(data, bits, precision=case["precision"])
            n = sum(k for cc, k in reqs if cc == c)
            st["models"].append(m)
            st["kept"].append(kept)
            st["X"].append(data.rows(n, 3).cpu().pin_memory())
            st["out"].append((torch.zeros(n, m.code_bytes, dtype=torch.uint8).pin_memory(),
                              torch.zeros(n, m.factor_count).pin_memory()))
        at = [0, 0, 0]
        st["reqs"] = []
        for c, n in reqs:
            st["reqs"].append((c, at[c], at[c] + n))
            at[c] += n
        st["service"] = P.Ingest(st["models"], hbm_budget_bytes=40 << 30, max_batch_rows=65536, slots=4)
        return st
    data = _Data(case["d"], case["alpha"], seed)
    if kind == "fit":
        st["X"] = data.rows(case["n"], 3)
        return st
    m, st["kept"] = _model(data, case["bits"], case.get("rounds", 6), case.get("precision", "fp32"))
    st["model"] = m
    X = data.rows(case["n"], 3)
    if kind == "encode":
        st["X"] = X
    elif kind == "encode_host":
        st["X"] = X.cpu().pin_memory()
        st["out"] = (torch.zeros(case["n"], max(m.code_bytes, 1), dtype=torch.uint8).pin_memory(),
                     torch.zeros(case["n"], m.factor_count).pin_memory())
    else:
        # a collection's codes and factors, and queries of the same distribution
        st["codes"], st["factors"] = m.encode(X)
        st["Q"] = data.rows(case["nq"], 5)
    return st


# ------------------------------------------------------------------- the call
def run(st):
    kind, case = st["kind"], st["case"]
    if kind == "encode":
        codes, factors = st["model"].encode(st["X"])
        return [codes, factors]
    if kind == "encode_host":
        codes, factors = st["model"].encode_host(st["X"], *st["out"])
        return [codes, factors]
    if kind == "serve":
        tickets = []
        for c, a, b in st["reqs"]:
            codes, factors = st["out"][c]
            tickets.append(st["service"].submit(c, st["X"][c][a:b], codes[a:b], factors[a:b]))
        for t in tickets:
            st["service"].wait(t)
        return [x for out in st["out"] for x in out]
    if kind == "estimate":
        return st["model"].estimate_dist(st["codes"], st["factors"], st["Q"], prefix_bits=case["prefix"])
    if kind == "staged":
        return st["model"].estimate_staged(st["codes"], st["factors"], st["Q"], case["m_conf"])
    m = P.saq_fit(st["X"], avg_bits=case["bits"])
    return {"mean": m.mean, "matrix": m.matrix, "variances": m.variances,
            "plan": np.array(m.plan, dtype=np.int64)}


# ------------------------------------------------------- what cannot be spared
def _plan_sizes(d, alpha, bits):
    """Kept dimensions, code bytes and factors of a model."""
    lam = np.arange(1, d + 1, dtype=np.float64) ** -alpha
    plan, _ = P.saq_plan_search(lam, int(round(bits * d)))
    kept = [(l, b) for _, l, b in plan if b > 0]
    return (sum(l for l, _ in kept), sum(b * ((l + 63) // 64) * 8 for l, b in kept), 1 + 2 * len(kept))


def work(case):
    kind = case["kind"]
    if kind == "serve":
        total = {"bytes": 0.0, "flops": 0.0}
        for c, (d, bits) in enumerate(_COLLECTIONS):
            n = sum(k for cc, k in _serve_sizes(case) if cc == c)
            w = work(dict(kind="encode", n=n, d=d, alpha=case["alpha"], bits=bits))
            total = {k: total[k] + w[k] for k in total}
        return total
    n, d = case["n"], case["d"]
    if kind == "fit":
        # the rows once, the covariance (its upper triangle) and the eigenvectors
        return {"bytes": 4.0 * n * d + 8.0 * d * d, "flops": n * d * (d + 1.0) + 9.0 * d ** 3}
    dk, cb, nf = _plan_sizes(d, case["alpha"], case["bits"])
    if kind in ("encode", "encode_host"):
        return {"bytes": n * (4.0 * d + cb + 4.0 * nf) + 4.0 * dk * d, "flops": 2.0 * n * d * dk}
    nq = case["nq"]
    out = 1 if kind == "estimate" else (nf - 1) // 2 + 1
    if case.get("prefix"):
        lam = np.arange(1, d + 1, dtype=np.float64) ** -case["alpha"]
        plan, _ = P.saq_plan_search(lam, int(round(case["bits"] * d)))
        cb = sum(min(b, case["prefix"]) * ((l + 63) // 64) * 8 for _, l, b in plan if b > 0)
    return {"bytes": n * (cb + 4.0 * nf) + 4.0 * nq * d + 4.0 * dk * d + 4.0 * nq * n * out,
            "flops": 2.0 * nq * n * dk + 2.0 * nq * d * dk * (1 if kind == "estimate" else 2)}


# ------------------------------------------------------------------ in 64 bits
def _factors64(X, kept):
    """Factors of rows X: |x - c|^2, and |o| and the cosine per kept segment
    after Algorithm 1 (initial codes, then the rounds of +1 / -1 trials)."""
    n = X.shape[0]
    out = torch.empty(n, 1 + 2 * len(kept.segs), dtype=F64, device="cuda")
    Xc = X.cuda().double() - kept.mean
    out[:, 0] = (Xc * Xc).sum(1)
    Ot = kept.W @ Xc.T  # one row per kept column
    del Xc
    off = 0
    for k, (_, length, b) in enumerate(kept.segs):
        O = Ot[off:off + length]
        off += length
        cmax = 2 ** b - 1
        v = O.abs().amax(0)
        live = v > 0
        delta = torch.where(live, 2 * v / 2 ** b, torch.ones_like(v))
        U = 2 * torch.clamp(torch.floor((O + v) / delta), 0, cmax) - cmax
        I, S = (U * O).sum(0), (U * U).sum(0)
        for _ in range(kept.rounds):
            moved = False
            for i in range(length):
                o, u = O[i], U[i]
                up = o * S > u * I  # the side the cosine can gain on
                s = torch.where(up, 1.0, -1.0).to(F64)
                In, Sn = I + 2 * s * o, S + 4 * s * u + 4
                ok = (s * u < cmax) & (In * S.sqrt() > I * Sn.sqrt()) & live
                U[i] = torch.where(ok, u + 2 * s, u)
                I, S = torch.where(ok, In, I), torch.where(ok, Sn, S)
                moved = ok.any() if moved is False else moved | ok.any()
            if not bool(moved):
                break
        nrm = O.square().sum(0).sqrt()
        one = torch.ones_like(nrm)
        out[:, 1 + 2 * k] = nrm
        out[:, 2 + 2 * k] = torch.where(live, I / (S.sqrt() * torch.where(live, nrm, one)), one)
    return out


def _decode(codes, length, b, off, prefix):
    """u of one segment (rows x length) from its bit-planes, most significant first."""
    words = (length + 63) // 64
    take = min(b, prefix) if prefix else b
    shift = torch.arange(8, device=codes.device)
    c = torch.zeros(codes.shape[0], length, dtype=torch.int64, device=codes.device)
    for p in range(take):
        plane = codes[:, off + p * words * 8:off + (p + 1) * words * 8].long()
        c = 2 * c + ((plane[:, :, None] >> shift) & 1).reshape(codes.shape[0], -1)[:, :length]
    return (2 * c - (2 ** take - 1)).double()


def _estimates64(st, staged):
    kept, codes, fac = st["kept"], st["codes"], st["factors"].double()
    prefix = st["case"].get("prefix", 0)
    Qc = st["Q"].double() - kept.mean
    q2, qr = (Qc * Qc).sum(1), Qc @ kept.W.T
    nq, n, nk = Qc.shape[0], codes.shape[0], len(kept.segs)
    res = torch.empty((nq, n, nk + 1) if staged else (nq, n), dtype=F64, device="cuda")
    sig = []
    if staged:
        pc = Qc @ kept.basis.T * kept.sigma
        at = 0
        for _, length, _ in kept.segs:
            sig.append(pc[:, at:at + length].square().sum(1).sqrt())
            at += length
    for i in range(0, n, 65536):
        j = min(n, i + 65536)
        base = fac[i:j, 0][None, :] + q2[:, None]
        done, at, cat = torch.zeros_like(base), 0, 0
        rest = [st["case"]["m_conf"] * sum(sig[t:], torch.zeros_like(q2))[:, None] for t in range(nk + 1)] if staged else None
        if staged:
            res[:, i:j, 0] = base - 2 * rest[0]
        for k, (_, length, b) in enumerate(kept.segs):
            u = _decode(codes[i:j], length, b, cat, prefix)
            nrm, cos = fac[i:j, 1 + 2 * k], fac[i:j, 2 + 2 * k]
            scale = torch.where(nrm > 0, nrm / (u.square().sum(1).sqrt() * cos), torch.zeros_like(nrm))
            done = done + (qr[:, at:at + length] @ u.T) * scale[None, :]
            at += length
            cat += b * ((length + 63) // 64) * 8
            if staged:
                res[:, i:j, k + 1] = base - 2 * (done + rest[k + 1])
        if not staged:
            res[:, i:j] = base - 2 * done
    return res


def exact(case, seed):
    kind = case["kind"]
    st = prepare(case, seed)
    if kind in ("encode", "encode_host"):
        return [None, _factors64(st["X"], st["kept"])]
    if kind == "serve":
        return [x for X, kept in zip(st["X"], st["kept"]) for x in (None, _factors64(X, kept))]
    if kind in ("estimate", "staged"):
        return _estimates64(st, kind == "staged")
    X = st["X"].double()
    mean = X.mean(0)
    Xc = X - mean
    var = torch.linalg.eigvalsh(Xc.T @ Xc / len(X)).flip(0).clamp_min(0)
    return {"mean": mean, "matrix": None, "variances": var, "plan": None}
