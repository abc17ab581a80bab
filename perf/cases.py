"""The work that users of this library have it do, as measurable cases: fused Langevin runs from single
short calls to resident-wave and streamed sizes, fills, batched systems, the adjoint and the overdamped
run, for every generator.  Each goes through the Python entry points of paper_1003_1123_gb300.gbrng.

A case names its path ("ld", "fill", "batched", "adjoint", "ou"), the generator and the sizes.  exact()
evaluates the same runs in 64 bits with plain torch: the integer streams by their definitions, the
uniforms' rounding to binary32 (which the definitions prescribe) and everything after it in binary64.
"""
import math

import numpy as np
import torch

from paper_1003_1123_gb300 import gbrng as G

DEV = "cuda"

# The paper's oscillator (Sec. IV test as configured here) and its overdamped particle.
LD = dict(m=1.0, gamma=0.5, kT=1.0, dt=0.01)
OU = dict(k_sp=0.01, xi=16.568, kT=4.142, dt=1.0)      # pN/nm, pN ps/nm, pN nm, ps; tau = xi/k_sp
KT_OVER_K = OU["kT"] / OU["k_sp"]


def listed():
    return [
        # a monitoring loop: a few steps, read the energies, decide, go on
        dict(name="ld_taus_short", path="ld", kind="taus", n=1000, steps=10, per_k=False),
        # the parity configuration, an ordinary small run
        dict(name="ld_taus_4096", path="ld", kind="taus", n=4096, steps=1000, per_k=False),
        # the throughput configuration (10^6 oscillators), a tenth of its steps
        dict(name="ld_taus_1e6", path="ld", kind="taus", n=10**6, steps=1000, per_k=False),
        # an odd mid-sized system with its own spring constants, the table generator
        dict(name="ld_ran2_100003", path="ld", kind="ran2", n=100003, steps=1000, per_k=True),
        # the shared generator at the paper's system size
        dict(name="ld_lagfib_1e4", path="ld", kind="lagfib", n=10**4, steps=1000, per_k=False),
        # the shared generator at the throughput configuration
        dict(name="ld_lagfib_1e6", path="ld", kind="lagfib", n=10**6, steps=1000, per_k=False),
        # the parity configuration's raw stream: 2^20 words of 4096 streams
        dict(name="fill_u32_taus", path="fill", op="u32", kind="taus", streams=4096, n=2**20),
        # normals for a host application, many streams, the table generator (an eighth of 2^30)
        dict(name="fill_normal_ran2", path="fill", op="normal", kind="ran2", streams=10**6, n=2**27),
        # uniforms from the shared sequence, odd length (a quarter of 2^30)
        dict(name="fill_uniform_lagfib", path="fill", op="uniform", kind="lagfib", streams=10**6,
             n=2**28 + 1),
        # the batched configuration: 512 uneven systems in one launch, a tenth of its steps
        dict(name="batched_taus_512", path="batched", kind="taus", systems=512, n_lo=100, n_hi=100000,
             shape_seed=1234, steps=500),
        # gradients of the averaged energy, checkpoints every 100 steps, a tenth of the steps
        dict(name="adjoint_taus_1e5", path="adjoint", kind="taus", n=10**5, steps=1000, ckpt=100),
        # the paper's overdamped test: 10^4 particles, <R(t)> and <R(t)R(0)> recorded
        dict(name="ou_taus_1e4", path="ou", kind="taus", n=10**4, steps=1000, every=100),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    path = rng.choice(["ld", "ld", "ld", "fill", "fill", "batched", "adjoint", "ou"])
    if path == "ld":
        n = _log_int(rng, 1000, 10**7)
        steps = _log_int(rng, 10, max(11, min(1000, 10**9 // n)))
        return dict(path=path, kind=rng.choice(["taus", "ran2", "lagfib", "lcg"]), n=n, steps=steps,
                    per_k=rng.random() < 0.5)
    if path == "fill":
        op = rng.choice(["u32", "uniform", "normal"])
        n = _log_int(rng, 2**16, 2**28)
        return dict(path=path, op=op, kind=rng.choice(["taus", "ran2", "lagfib", "lcg"]),
                    streams=_log_int(rng, 1024, 10**6), n=n & ~1 if op == "normal" else n)
    if path == "batched":
        n_hi = _log_int(rng, 1000, 100000)
        return dict(path=path, kind=rng.choice(["taus", "ran2"]), systems=_log_int(rng, 8, 512),
                    n_lo=100, n_hi=n_hi, shape_seed=rng.randrange(10**6), steps=_log_int(rng, 50, 500))
    if path == "adjoint":
        return dict(path=path, kind=rng.choice(["taus", "ran2"]), n=_log_int(rng, 1000, 10**5),
                    steps=_log_int(rng, 100, 1000), ckpt=rng.choice([50, 64, 100]))
    n = _log_int(rng, 1000, 10**6)
    steps = _log_int(rng, 100, min(5000, 10**9 // n))
    return dict(path=path, kind=rng.choice(["taus", "ran2", "lagfib", "lcg"]), n=n, steps=steps,
                every=max(1, steps // 10))


# --------------------------------------------------------------------- inputs
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def _rng_seed(seed):
    return (seed * 0x9E3779B97F4A7C15 + 12345) % 2**64


def _phase(n, seed, K, kT, m):
    """An equilibrium start: x ~ N(0, kT/K), v ~ N(0, kT/m)."""
    g = _gen(seed)
    x = torch.randn((n, 3), generator=g, device=DEV) * (kT / K).sqrt().reshape(-1, 1)
    v = torch.randn((n, 3), generator=g, device=DEV) * math.sqrt(kT / m)
    return x.contiguous(), v.contiguous()


def _spring(case, seed):
    n = case["n"]
    if case["path"] == "ld" and not case["per_k"]:
        return None, torch.ones(1, device=DEV)
    K = torch.rand(n, generator=_gen(seed + 1), device=DEV) * 1.5 + 0.5
    return K, K


def _batch(case):
    """Parameters of the systems: N log-uniform, K log-uniform in [0.1, 10], gamma in [0.1, 2], kT in
    [0.5, 2] (a program keeps its systems; their states come from the seed)."""
    r = np.random.default_rng(case["shape_seed"])
    S = case["systems"]
    n = np.exp(r.uniform(np.log(case["n_lo"]), np.log(case["n_hi"]), S)).astype(np.int64)
    K = np.exp(r.uniform(np.log(0.1), np.log(10.0), S))
    return n, K, r.uniform(0.1, 2.0, S), r.uniform(0.5, 2.0, S)


def _batch_start(case, seed):
    n, K, gamma, kT = _batch(case)
    per = torch.from_numpy(np.repeat(np.sqrt(kT / K), n)).to(DEV, torch.float32).reshape(-1, 1)
    perv = torch.from_numpy(np.repeat(np.sqrt(kT), n)).to(DEV, torch.float32).reshape(-1, 1)
    g = _gen(seed)
    total = int(n.sum())
    x = torch.randn((total, 3), generator=g, device=DEV) * per
    v = torch.randn((total, 3), generator=g, device=DEV) * perv
    return x, v


def _ou_start(case, seed):
    return torch.randn(case["n"], generator=_gen(seed), device=DEV) * math.sqrt(KT_OVER_K)


def prepare(case, seed):
    path = case["path"]
    if path == "fill":
        return dict(case, rng=G.rng_init(case["kind"], _rng_seed(seed), case["streams"]))
    if path == "batched":
        n, K, gamma, kT = _batch(case)
        x, v = _batch_start(case, seed)
        cut = np.concatenate([[0], np.cumsum(n)])
        systems = []
        for s in range(case["systems"]):
            rng = G.rng_init(case["kind"], _rng_seed(seed) ^ s, int(n[s]))
            systems.append(G.LdSystem(rng, x[cut[s]:cut[s + 1]], v[cut[s]:cut[s + 1]], K=K[s], m=1.0,
                                      gamma=gamma[s], kT=kT[s], dt=0.005))
        return dict(case, systems=systems, x=x, v=v)
    rng = G.rng_init(case["kind"], _rng_seed(seed), case["n"])
    if path == "ou":
        return dict(case, system=G.OuSystem(rng, _ou_start(case, seed), **OU))
    K_per, K = _spring(case, seed)
    x, v = _phase(case["n"], seed, K, LD["kT"], LD["m"])
    return dict(case, system=G.LdSystem(rng, x, v, K=1.0, K_per=K_per, **LD))


# ----------------------------------------------------------------------- runs
_FILL = {"u32": G.rng_fill_u32, "uniform": G.rng_fill_uniform, "normal": G.rng_fill_normal}


def run(state):
    path = state["path"]
    if path == "fill":
        return _FILL[state["op"]](state["rng"], state["n"])
    if path == "ld":
        s = state["system"]
        st = G.ld_run(s, state["steps"])
        return {"x": s.x, "v": s.v, "stats": st}
    if path == "batched":
        st = G.ld_run_batched(state["systems"], state["steps"])
        return {"x": state["x"], "v": state["v"],
                "energy": np.array([s["energy_time_avg"] for s in st], np.float32)}
    if path == "adjoint":
        s = state["system"]
        r = G.ld_backward(s, state["steps"], state["ckpt"])
        return {"x": s.x, "v": s.v, **r}
    s = state["system"]
    mean, corr = G.ou_run(s, state["steps"], state["every"])
    return {"R": s.R, "mean": mean, "corr": corr}


# ----------------------------------------------------------------------- work
# Operations of one draw as the algorithms print them (shifts, logic, multiplies, adds), and of the
# transform and the updates, an elementary function as one.
_DRAW = {"taus": 23, "ran2": 15, "lcg": 2, "lagfib": 2}
_NORMALS3 = 4 * 2 + 2 * 5 + 1          # four uniforms, two transforms, the second sine dropped
_STEP = 3 * 6 + 14                     # update of three components, energy


def _state_bytes(kind, streams):
    if kind == "lagfib":
        return 4 * G.rng_lfg_lags(G.rng_lfg_default_row(streams))[1]
    return {"taus": 16, "ran2": 140, "lcg": 4}[kind] * streams


def work(case):
    path, kind = case["path"], case["kind"]
    if path == "fill":
        active = case["streams"] if kind == "lagfib" else min(case["streams"], case["n"])
        per = {"u32": 0, "uniform": 2, "normal": 4}[case["op"]]
        return {"bytes": 4 * case["n"] + 2 * _state_bytes(kind, active),
                "flops": case["n"] * (_DRAW[kind] + per)}
    if path == "ou":
        n, steps = case["n"], case["steps"]
        return {"bytes": 8 * n + 2 * _state_bytes(kind, n) + 16 * (steps // case["every"] + 1),
                "flops": n * steps * (2 * _DRAW[kind] + 4 + 5 + 4)}
    n = int(_batch(case)[0].sum()) if path == "batched" else case["n"]
    per_k = 4 * n if path == "adjoint" or case.get("per_k") else 0
    step = 4 * _DRAW[kind] + _NORMALS3 + _STEP
    b = 48 * n + 2 * _state_bytes(kind, n) + per_k
    if path == "adjoint":
        b, step = b + 4 * n, step + 3 * 16 + 3
    return {"bytes": b, "flops": n * case["steps"] * step}


# ------------------------------------------------------------- 64-bit reference
_U32 = 0xFFFFFFFF


def _wrap64(c):
    c %= 2**64
    return c - 2**64 if c >= 2**63 else c


def _shr64(z, s):
    """Logical right shift of int64 words."""
    return (z >> s) & ((1 << (64 - s)) - 1)


def _splitmix(seed, idx):
    """SplitMix64 at counters idx (int64 tensor); int64 arithmetic wraps as uint64 does.  `seed`: an int
    or an int64 tensor of the same shape."""
    if not torch.is_tensor(seed):
        seed = _wrap64(seed)
    z = (idx + 1) * _wrap64(0x9E3779B97F4A7C15) + seed
    z = (z ^ _shr64(z, 30)) * _wrap64(0xBF58476D1CE4E5B9)
    z = (z ^ _shr64(z, 27)) * _wrap64(0x94D049BB133111EB)
    return z ^ _shr64(z, 31)


class _Streams:
    """Per-thread generators of a vector of streams: stream s[i] of the generator seeded seed[i]."""

    def __init__(self, kind, seed, stream):
        self.kind = kind
        word = lambda k: _splitmix(seed, stream * 8 + k)          # noqa: E731
        if kind == "taus":
            w = [word(k) & _U32 for k in range(4)]
            self.y = [torch.where(w[i] < f, w[i] + f, w[i]) for i, f in enumerate((2, 8, 16))] + [w[3]]
        elif kind == "lcg":
            self.x = word(0) & _U32
        else:
            w, m = word(0), 2147483562
            # unsigned 64-bit remainder from the two halves
            r = (_shr64(w, 32) % m * (2**32 % m) + (w & _U32) % m) % m
            self.idum = 1 + r
            self.idum2 = self.idum.clone()
            self.tab = torch.zeros((32,) + tuple(stream.shape), dtype=torch.int64, device=DEV)
            for j in range(39, -1, -1):
                self.idum = self.idum * 40014 % 2147483563
                if j < 32:
                    self.tab[j] = self.idum
            self.iy = self.tab[0].clone()

    def raw(self):
        if self.kind == "taus":
            y = self.y
            for i, (a, b, c, mask) in enumerate(((13, 19, 12, 4294967294), (2, 25, 4, 4294967288),
                                                 (3, 11, 17, 4294967280))):
                t = (((y[i] << a) & _U32) ^ y[i]) >> b
                y[i] = (((y[i] & mask) << c) & _U32) ^ t
            y[3] = (y[3] * 1664525 + 1013904223) & _U32
            return y[0] ^ y[1] ^ y[2] ^ y[3]
        if self.kind == "lcg":
            self.x = (self.x * 1664525 + 1013904223) & _U32
            return self.x
        self.idum = self.idum * 40014 % 2147483563
        self.idum2 = self.idum2 * 40692 % 2147483399
        j = (self.iy // (1 + 2147483562 // 32)).unsqueeze(0)
        y = self.tab.gather(0, j)[0] - self.idum2
        self.tab.scatter_(0, j, self.idum.unsqueeze(0))
        self.iy = torch.where(y < 1, y + 2147483562, y)
        return self.iy


class _Shared:
    """The shared Lagged Fibonacci sequence, generated in blocks of up to ll - sl values."""

    def __init__(self, seed, threads):
        self.sl, self.ll = G.rng_lfg_lags(G.rng_lfg_default_row(threads))
        w = torch.arange(self.ll, dtype=torch.int64, device=DEV)
        h = _splitmix(seed, w) & _U32
        h[0] |= 1
        self.hist = h.to(torch.int64)
        self.left = h[:0]

    def take(self, count):
        D = self.ll - self.sl
        got, have = [self.left], self.left.numel()
        while have < count:
            b = D if D < self.ll else self.ll
            new = (self.hist[:b] + self.hist[self.sl:self.sl + b]) & _U32
            self.hist = torch.cat([self.hist[b:], new])
            got.append(new)
            have += b
        all_ = torch.cat(got)
        self.left = all_[count:]
        return all_[:count]


def _uniform(kind, raw):
    """The binary32 uniform of a fill, in binary64."""
    if kind == "ran2":
        u = raw.to(torch.float32).double() * 2.0**-31
        return torch.clamp(u, max=1.0 - 2.0**-24)
    return raw.to(torch.float32).double() * 2.0**-32


def _open(kind, raw):
    """Box-Muller's input in (0, 1)."""
    if kind == "ran2":
        return _uniform(kind, raw)
    return ((raw >> 9).double() + 0.5) * 2.0**-23


def _pair(kind, r1, r2):
    rho = torch.sqrt(-2.0 * torch.log(_open(kind, r1)))
    a = 2.0 * math.pi * _open(kind, r2)
    return rho * torch.cos(a), rho * torch.sin(a)


def _source(case, seed, n):
    """A function giving the next `k` raw draws of n oscillators as k tensors [n]."""
    if case["kind"] == "lagfib":
        sh = _Shared(_rng_seed(seed), case["n"])
        return lambda k: list(sh.take(k * n).reshape(n, k).t().contiguous())
    st = _Streams(case["kind"], _rng_seed(seed), torch.arange(n, dtype=torch.int64, device=DEV))
    return lambda k: [st.raw() for _ in range(k)]


def _normals3(kind, r):
    g0, g1 = _pair(kind, r[0], r[1])
    g2, _ = _pair(kind, r[2], r[3])
    return torch.stack([g0, g1, g2], 1)


def _f32(v):
    return float(np.float32(v))


def _ld_coef(m, gamma, kT, dt):
    """The step's coefficients, rounded once to binary32 as the interface states."""
    return _f32(dt), _f32(1.0 - gamma * dt / m), _f32(dt / m), _f32(math.sqrt(2 * gamma * kT * dt) / m)


def _ld_exact(kind, draws, x, v, K, coef, m, steps):
    """(x, v, time-averaged energy per oscillator) after the steps; coef may hold [n, 1] tensors."""
    cdt, cva, ckm, cs = coef
    x, v, K = x.double(), v.double(), K.double().reshape(-1, 1)
    ck = ckm * K
    e = torch.zeros(x.shape[0], dtype=torch.float64, device=DEV)
    for _ in range(steps):
        g = _normals3(kind, draws(4))
        x, v = x + cdt * v, cva * v + (cs * g - ck * x)
        e += 0.5 * (m * v.square().sum(1) + K[:, 0] * x.square().sum(1))
    return x, v, e / steps


def exact(case, seed):
    path, kind = case["path"], case["kind"]
    if path == "fill":
        return _fill_exact(case, seed)
    if path == "batched":
        n, K, gamma, kT = _batch(case)
        per = lambda a: torch.from_numpy(np.repeat(a, n)).to(DEV)          # noqa: E731
        ids = np.concatenate([np.arange(k, dtype=np.int64) for k in n])
        seeds = np.array([_wrap64(_rng_seed(seed) ^ s) for s in range(len(n))], np.int64)
        st = _Streams(kind, per(seeds), torch.from_numpy(ids).to(DEV))
        x, v = _batch_start(case, seed)
        c = [_ld_coef(1.0, g, t, 0.005) for g, t in zip(gamma, kT)]
        coef = [per(np.array([q[i] for q in c])).reshape(-1, 1) for i in range(4)]
        K32 = per(K.astype(np.float32).astype(np.float64))
        x, v, e = _ld_exact(kind, lambda k: [st.raw() for _ in range(k)], x, v, K32, coef, 1.0,
                            case["steps"])
        out = torch.zeros(len(n), dtype=torch.float64, device=DEV)
        out.index_add_(0, per(np.arange(len(n))), e)
        return {"x": x, "v": v, "energy": out}
    n = case["n"]
    draws = _source(case, seed, n)
    if path == "ou":
        return _ou_exact(case, seed, draws)
    _, K = _spring(case, seed)
    x, v = _phase(n, seed, K, LD["kT"], LD["m"])
    K = K.expand(n)
    coef = _ld_coef(**LD)
    if path == "adjoint":
        return _adjoint_exact(case, draws, x, v, K, coef)
    x, v, e = _ld_exact(kind, draws, x, v, K, coef, LD["m"], case["steps"])
    stats = {"sum_x2": float((x * x).sum()), "sum_v2": float((v * v).sum()),
             "sum_xv": float((x * v).sum()), "energy_time_avg": float(e.sum()), "steps": case["steps"]}
    return {"x": x, "v": v, "stats": stats}


def _fill_exact(case, seed):
    kind, n, op = case["kind"], case["n"], case["op"]
    count = 1 if op != "normal" else 2
    if kind == "lagfib":
        raw = _Shared(_rng_seed(seed), case["streams"]).take(n)
        r = [raw] if count == 1 else [raw[0::2], raw[1::2]]
    else:
        # whole rows of one item a stream, then cut
        S, items = case["streams"], n // count
        st = _Streams(kind, _rng_seed(seed),
                      torch.arange(min(S, items), dtype=torch.int64, device=DEV))
        got = [[st.raw() for _ in range(count)] for _ in range(-(-items // S))] if items // S < 20000 else None
        if got is None:
            return None
        r = [torch.cat([g[k] for g in got])[:items] for k in range(count)]
    if op == "u32":
        return r[0].to(torch.int32)
    if op == "uniform":
        return _uniform(kind, r[0])
    return torch.stack(_pair(kind, *r), 1).reshape(-1)


def _ou_exact(case, seed, draws):
    R = _ou_start(case, seed).double()
    R0 = R.clone()
    c1 = _f32(OU["k_sp"] * OU["dt"] / OU["xi"])
    cs = _f32(math.sqrt(2 * OU["kT"] * OU["dt"] / OU["xi"]))
    mean, corr = [], []
    for t in range(case["steps"] + 1):
        if t % case["every"] == 0:
            mean.append(float(R.mean()))
            corr.append(float((R * R0).mean()))
        if t < case["steps"]:
            g, _ = _pair(case["kind"], *draws(2))
            R = R - c1 * R + cs * g
    return {"R": R, "mean": np.array(mean), "corr": np.array(corr)}


def _adjoint_exact(case, draws, x, v, K, coef):
    """The discrete adjoint of L = (1/S) sum_t E(t) over the stored trajectory."""
    cdt, cva, ckm, cs = coef
    S, m, gamma, kT = case["steps"], LD["m"], LD["gamma"], LD["kT"]
    x, v, K = x.double(), v.double(), K.double().reshape(-1, 1)
    ck = ckm * K
    path, loss, xsq = [], 0.0, 0.0
    for _ in range(S):
        g = _normals3(case["kind"], draws(4))
        path.append((x, v, g))
        x, v = x + cdt * v, cva * v + (cs * g - ck * x)
        loss = loss + 0.5 * (m * v.square().sum() + (K * x.square()).sum())
        xsq = xsq + x.square().sum(1)
    lx, lv = K * x / S, m * v / S
    dK = 0.5 * xsq / S
    dg = dT = 0.0
    for t in range(S - 1, -1, -1):
        xt, vt, g = path[t]
        dK = dK - ckm * (lv * xt).sum(1)
        dg = dg + (lv * (cs / (2 * gamma) * g - ckm * vt)).sum()
        dT = dT + (lv * g).sum() * (cs / (2 * kT))
        w = 1.0 / S if t else 0.0
        lx, lv = lx - ck * lv + w * K * xt, cdt * lx + cva * lv + w * m * vt
    return {"x": x, "v": v, "loss": float(loss) / S, "dgamma": float(dg), "dkT": float(dT), "dK": dK}
