"""What a user of this package has it compute, as measurable passes.

Each case is one call (or one short program) through the public binding
``paper_1612_09517_gb300.rp``: singlet yields over a field sweep, a batch of
uneven radical pairs, time-resolved observables, one H psi, and the control
variate's inference.  The nuclei, rates, exchange, field ranges and precisions
are those of the seeded workloads in ``paper_1612_09517_gb300/workloads.py``;
horizons and sample counts are cut so that a pass takes a fraction of a second
(the work per Chebyshev term and row is unchanged by that).  A seed gives other
hyperfine couplings and other samples of the same distributions.

Yields are averages of wavepacket propagations in the precision the caller asks
for; the C ABI returns them in FP64 arrays.  ``run`` returns the results of an
FP32 call as FP32 arrays, the precision they carry, and those of an FP64 call
as FP64 arrays.
"""
import math

import numpy as np
import torch

from paper_1612_09517_gb300 import rp
from paper_1612_09517_gb300 import workloads as wl

GAMMA_E = 176.085963023  # |gamma_e|, rad us^-1 mT^-1 (CODATA 2018)
N_CHEB = 88              # default Chebyshev terms per macro-step


def _case(name, kind, half=(0, 0), one=(0, 0), big=(0, 0), aniso=False, J=0.0, k_S=1.0, k_T=1.0,
          precision="fp32", n_fields=1, B_max=10.0, M=2, T=1.0, deterministic=0, **more):
    """half / one / big: spin-1/2, spin-1 and spin-3/2 nuclei on radical 1 and radical 2."""
    c = dict(kind=kind, half1=half[0], half2=half[1], one1=one[0], one2=one[1], big1=big[0],
             big2=big[1], aniso=aniso, J=J, k_S=k_S, k_T=k_T, precision=precision,
             n_fields=n_fields, B_max=B_max, M=M, T=T, deterministic=deterministic, **more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one H psi of a few states of a four-nucleus pair: a user's own propagator
        # or a check against another code; the call is all latency
        _case("apply_h_small", "apply", half=(4, 0), k_S=1.0, k_T=1.0, precision="fp64", M=16),
        # a quick look at one field of a small pair (six nuclei, one of them spin-1)
        _case("one_field_z96", "yields", half=(3, 2), one=(0, 1), k_S=2.0, k_T=0.5, n_fields=1,
              B_max=3.0, M=16, T=5.0),
        # the four-nucleus sweep in full (11 fields in 0-5 mT, M = 64, 10 us), in FP64
        _case("sweep_z16_fp64", "yields", half=(4, 0), precision="fp64", n_fields=11, B_max=5.0,
              M=64, T=10.0),
        # a pair of the 256-pair ensemble whose state fits one SM (Z = 864)
        _case("sweep_z864", "yields", half=(3, 2), one=(1, 2), k_S=1.5, k_T=0.4, n_fields=32,
              B_max=10.0, M=32, T=2.0),
        # a pair of the ensemble between one SM and the 12-nucleus workload (Z = 4608)
        _case("sweep_z4608", "yields", half=(5, 4), one=(1, 1), k_S=0.8, k_T=3.0, n_fields=16,
              B_max=10.0, M=8, T=2.0),
        # the headline workload: 12 nuclei, Z = 20736, 32 fields in 0-50 mT x 2 samples (one
        # step of the benchmark)
        _case("sweep_z20736", "yields", half=(5, 3), one=(2, 2), k_S=2.0, k_T=0.5, n_fields=32,
              B_max=50.0, M=2, T=0.25),
        # the same pair in FP64, the form used to check a curve
        _case("sweep_z20736_fp64", "yields", half=(5, 3), one=(2, 2), k_S=2.0, k_T=0.5,
              precision="fp64", n_fields=8, B_max=50.0, M=2, T=0.05),
        # 20 nuclei with anisotropic tensors and exchange, Z = 2359296
        _case("aniso_z2359296", "yields", half=(9, 9), one=(1, 1), aniso=True, J=0.1, n_fields=3,
              B_max=10.0, M=2, T=0.06),
        # the paper's 20 spin-1/2 model problem, Z = 2^20, J = 1.75 mT
        _case("table1_z1048576", "yields", half=(10, 10), J=1.75, k_S=17.6, k_T=176.0,
              n_fields=7, B_max=10.0, M=2, T=0.08),
        # a batch of uneven pairs of the ensemble in one call
        _case("batch_uneven", "batch", n_fields=4, B_max=10.0, M=4, T=0.3, n_pairs=12, n_max=12,
              z_max=30000, mix=1004),
        # P_S(t), P_T(t) and survival of an anisotropic pair in FP64
        _case("trace_aniso_z192_fp64", "trace", half=(3, 3), one=(1, 0), aniso=True, J=0.1,
              precision="fp64", B_max=2.0, M=32, T=2.0),
        # the control variate's E[g] over fresh directions and g of the samples in hand
        _case("cv_inference", "cv", half=(5, 3), one=(2, 2), n_fields=8, B_max=10.0, M=4096,
              n_mc=65536, hidden=256, layers=3),
    ]


# ---- inputs (pure NumPy: the same for run and exact) ----

def _radical_two_I(c):
    two_I, radical = [], []
    for r in (0, 1):
        s = [1] * c[f"half{r + 1}"] + [2] * c[f"one{r + 1}"] + [3] * c[f"big{r + 1}"]
        two_I += s
        radical += [r] * len(s)
    return radical, two_I


def _tensors(rng, n, aniso):
    A = np.empty((n, 3, 3))
    for k in range(n):
        if aniso:
            q, _ = np.linalg.qr(rng.normal(size=(3, 3)))
            A[k] = q @ np.diag(rng.normal(0.0, 0.8, 3)) @ q.T
            A[k] = 0.5 * (A[k] + A[k].T)
        else:
            A[k] = rng.normal(0.0, 0.5) * np.eye(3)
    return A


def _fields(c):
    return np.linspace(0.0, c["B_max"], c["n_fields"]) if c["n_fields"] > 1 else np.array([c["B_max"]])


def _batch_shapes(c):
    """Nuclei and rates of the pairs of a batch: the ensemble's distributions, by `mix` alone."""
    rng = np.random.default_rng(c["mix"])
    out = []
    while len(out) < c["n_pairs"]:
        n = int(rng.integers(6, c["n_max"] + 1))
        two_I = np.where(rng.uniform(size=n) < 0.8, 1, 2)
        k = 10.0 ** rng.uniform(-1.0, 1.0, 2)
        if np.prod(two_I + 1.0) <= c["z_max"]:
            n1 = (n + 1) // 2
            out.append(([0] * n1 + [1] * (n - n1), [int(t) for t in two_I], float(k[0]), float(k[1]),
                        c["T"] / float(max(k.min(), 0.3))))
    return out


def _inputs(c, seed):
    """The pairs of the call: a list of (SpinSystem, horizon)."""
    # (a time trace keeps its pair, and with it the number of time points, for every seed)
    rng = np.random.default_rng([0 if c["kind"] == "trace" else seed, 77])
    if c["kind"] == "batch":
        return [(wl.SpinSystem(r, t, _tensors(rng, len(t), c["aniso"]), kS, kT, 0.0), T)
                for r, t, kS, kT, T in _batch_shapes(c)]
    r, t = _radical_two_I(c)
    return [(wl.SpinSystem(r, t, _tensors(rng, len(t), c["aniso"]), c["k_S"], c["k_T"], c["J"]), c["T"])]


def _apply_vectors(c, Z, seed):
    rng = np.random.default_rng([seed, 78])
    x = rng.normal(size=(c["M"], 4 * Z, 2))
    return (x / np.sqrt((x ** 2).sum(axis=(1, 2), keepdims=True))).astype(_real(c))


def _cv_params(c, d_in, seed):
    """He-scaled weights and small biases, flat (W_0, b_0, W_1, b_1, ...)."""
    rng = np.random.default_rng([seed, 79])
    dims = [d_in] + [c["hidden"]] * c["layers"] + [1]
    parts = []
    for a, b in zip(dims[:-1], dims[1:]):
        parts += [rng.uniform(-1, 1, b * a) * math.sqrt(6.0 / a), rng.uniform(-0.1, 0.1, b)]
    return np.concatenate(parts).astype(np.float32), dims


def _real(c):
    return np.float64 if c["precision"] == "fp64" else np.float32


# ---- the calls ----

def prepare(case, seed):
    torch.cuda.set_device(0)
    rp.use_torch_allocator()
    c = dict(case)
    pairs = _inputs(c, seed)
    st = {"c": c, "seed": seed, "systems": [rp.System(s) for s, _ in pairs],
          "T": [t for _, t in pairs], "fields": _fields(c),
          "opt": rp.rp_default_options(precision=c["precision"], deterministic=c["deterministic"])}
    sy = st["systems"][0]
    if c["kind"] == "apply":
        st["x"] = torch.from_numpy(_apply_vectors(c, sy.Z, seed)).cuda()
        st["y"] = torch.empty_like(st["x"])
    elif c["kind"] == "cv":
        st["cv"] = rp.ControlVariate(sy, hidden=c["hidden"], layers=c["layers"])
        st["cv"].set_params(_cv_params(c, st["cv"].d_in, seed)[0])
        st["B"] = np.resize(st["fields"], c["M"])
        st["samples"] = np.arange(c["M"], dtype=np.int64)
    return st


def run(state):
    c, sy, opt = state["c"], state["systems"][0], state["opt"]
    f = _real(c)
    if c["kind"] == "yields":
        r = rp.rp_yields(sy.handle, state["fields"], c["M"], state["seed"], c["T"], opt,
                         per_sample=True)
        return {"out": r["out"].astype(f), "per_sample": r["per_sample"].astype(f)}
    if c["kind"] == "batch":
        n = len(state["systems"])
        r = rp.rp_yields_batch(state["systems"], [state["fields"]] * n, [c["M"]] * n, state["T"],
                               state["seed"], opt)
        return {"out": np.stack(r["out"]).astype(f)}
    if c["kind"] == "trace":
        t, o = rp.rp_time_trace(sy.handle, c["B_max"], c["M"], state["seed"], c["T"], opt)
        return {"t": t, "out": o.astype(f)}
    if c["kind"] == "apply":
        rp.rp_apply_h(sy.handle, c["B_max"], opt.precision, c["M"], state["x"].data_ptr(),
                      state["y"].data_ptr(), torch.cuda.current_stream().cuda_stream)
        return {"y": state["y"]}
    mu, var_mu = state["cv"].mean(state["fields"], c["n_mc"], state["seed"])
    g = state["cv"].eval(state["B"], state["samples"], state["seed"])
    return {"mu": mu.astype(f), "var_mu": var_mu.astype(f), "g": g.astype(f)}


# ---- what a pass cannot do without ----

def _mean_range(c, two_I):
    """Expected half-width (mT) of the hyperfine spectrum, summed over the nuclei."""
    one = {1: 0.5, 2: 0.75, 3: 1.0}
    return sum(one[t] * (1.1 if c["aniso"] else 0.4) for t in two_I)


def _terms(c, two_I, B, T):
    """Chebyshev terms of one propagation: N_CHEB per macro-step of dE h = 46 (FP64) or 56 (FP32)."""
    dE = GAMMA_E * (abs(B) + _mean_range(c, two_I) + abs(c["J"]))
    return N_CHEB * max(1, math.ceil(dE * T / (46.0 if c["precision"] == "fp64" else 56.0)))


def _term_flops(c, two_I):
    """Per nuclear configuration and term: H psi (Eq. 1), the recurrence, psi(h) and the time integral."""
    partners = sum(2.0 * t / (t + 1.0) for t in two_I)
    return partners * (24.0 if c["aniso"] else 8.0) + (80.0 if c["aniso"] else 40.0) + 16.0 + 32.0 + 120.0


def work(case):
    c = dict(case)
    size = 8 if c["precision"] == "fp64" else 4
    if c["kind"] == "cv":
        d = 3 * len(_radical_two_I(c)[1]) + 10
        per = 2.0 * (d * c["hidden"] + (c["layers"] - 1) * c["hidden"] ** 2 + c["hidden"])
        n = c["n_fields"] * c["n_mc"] + c["M"]
        return {"bytes": 16.0 * c["M"] + 4.0 * c["M"], "flops": per * n}
    if c["kind"] == "batch":
        shapes = [(t, T) for _, t, _, _, T in _batch_shapes(c)]
    else:
        shapes = [(_radical_two_I(c)[1], c["T"])]
    flops = nbytes = 0.0
    for two_I, T in shapes:
        Z = float(np.prod(np.array(two_I) + 1.0)) if two_I else 1.0
        if c["kind"] == "apply":
            flops += c["M"] * Z * (_term_flops(c, two_I) - 168.0)
            nbytes += 2.0 * c["M"] * Z * 8 * size
            continue
        rows = Z if c["deterministic"] == 1 else c["M"]
        for B in _fields(c):
            n = _terms(c, two_I, B, T) * rows
            flops += n * Z * _term_flops(c, two_I)
            nbytes += rows * 24.0
            if 2 * Z * 8 * size > 128e6:
                # two vectors of a row exceed the L2: each term reads phi_{n-1} and
                # phi_{n-2} from memory and writes phi_n
                nbytes += 3.0 * n * Z * 8 * size
    return {"bytes": nbytes, "flops": flops}


# ---- drawn cases ----

def _cost(c):
    """Work in FP32 flops of this chip (FP64 runs at 1/64 of the FP32 rate)."""
    return work(c)["flops"] * (64.0 if c["precision"] == "fp64" and c["kind"] != "cv" else 1.0)


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_nuclei(rng, z_max):
    """Nuclei of one pair: log2 Z uniform up to z_max, spins as in the ensemble, a few spin-3/2."""
    target = rng.uniform(1.0, math.log2(z_max))
    n = {(s, r): 0 for s in (1, 2, 3) for r in (0, 1)}
    z = 0.0
    while True:
        s = rng.choices((1, 2, 3), weights=(0.78, 0.2, 0.02))[0]
        if z + math.log2(s + 1) > target or sum(n.values()) >= 24:
            break
        z += math.log2(s + 1)
        n[(s, rng.randrange(2))] += 1
    return dict(half=(n[1, 0], n[1, 1]), one=(n[2, 0], n[2, 1]), big=(n[3, 0], n[3, 1]))


def draw(rng):
    cap = 0.5 * max(_cost(c) for c in listed())
    kind = rng.choices(("yields", "batch", "trace", "apply", "cv"), weights=(12, 2, 2, 1, 1))[0]
    prec = "fp64" if rng.random() < 0.3 else "fp32"
    k = [round(10.0 ** rng.uniform(-1.0, 1.0), 3) for _ in range(2)]
    common = dict(precision=prec, k_S=k[0], k_T=k[1], B_max=round(rng.uniform(0.5, 50.0), 2))
    if kind == "cv":
        return _case("", "cv", **{**_draw_nuclei(rng, 1 << 16)}, B_max=10.0,
                     n_fields=rng.randint(1, 8), M=_log_int(rng, 16, 20000),
                     n_mc=_log_int(rng, 2000, 65536), hidden=rng.choice((64, 128, 200, 256)),
                     layers=rng.randint(2, 3))
    if kind == "batch":
        c = _case("", "batch", **{**common, "B_max": 10.0}, n_fields=rng.randint(1, 6),
                  M=rng.randint(2, 8), T=round(rng.uniform(0.1, 0.5), 3), n_pairs=rng.randint(2, 24),
                  n_max=rng.randint(7, 12), z_max=30000, mix=rng.randrange(1 << 20))
    elif kind == "apply":
        return _case("", "apply", **common, **_draw_nuclei(rng, 1 << 20), aniso=rng.random() < 0.4,
                     J=rng.choice((0.0, 0.3)), M=rng.randint(1, 16))
    else:
        aniso = rng.random() < 0.3
        nuclei = _draw_nuclei(rng, 1 << (14 if prec == "fp64" else 20))
        c = _case("", kind, **common, **nuclei, aniso=aniso, J=rng.choice((0.0, 0.0, 0.1, 1.75)),
                  n_fields=1 if kind == "trace" else _log_int(rng, 1, 64), M=_log_int(rng, 2, 64),
                  T=round(math.exp(rng.uniform(math.log(0.05), math.log(10.0))), 4))
    # the horizon, then samples and fields, give way where the call would cost too much
    while _cost(c) > cap:
        if c["T"] > 0.02:
            c["T"] = round(0.7 * c["T"], 5)
        elif c["M"] > 2:
            c["M"] = max(2, c["M"] // 2)
        elif c["n_fields"] > 1:
            c["n_fields"] //= 2
        else:
            break
    return c


# ---- the same quantities in 64 bits, from the formulas alone (torch and NumPy) ----

def _philox(seed, pair, samples, n_nuc):
    """Uniforms (u1, u2) of Philox4x32-10 with counter (nucleus, s_lo, s_hi, pair) and key seed."""
    m0, m1, mask = 0xD2511F53, 0xCD9E8D57, np.uint64(0xFFFFFFFF)
    s = np.asarray(samples, dtype=np.uint64)[:, None]
    k = np.arange(n_nuc, dtype=np.uint64)[None, :]
    c = [np.broadcast_to(v, (s.size, n_nuc)).copy() for v in
         (k, s & mask, s >> np.uint64(32), np.uint64(pair))]
    k0, k1 = seed & 0xFFFFFFFF, seed >> 32
    for _ in range(10):
        p0, p1 = c[0] * np.uint64(m0), c[2] * np.uint64(m1)
        c = [(p1 >> np.uint64(32)) ^ c[1] ^ np.uint64(k0), p1 & mask,
             (p0 >> np.uint64(32)) ^ c[3] ^ np.uint64(k1), p0 & mask]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF

    def u53(hi, lo):
        return ((hi >> np.uint64(5)).astype(float) * 2.0 ** 26 + (lo >> np.uint64(6)).astype(float)) / 2.0 ** 53
    return u53(c[0], c[1]), u53(c[2], c[3])


def _spin(two_I):
    d = two_I + 1
    M = 0.5 * two_I - np.arange(d)
    up = np.diag(np.sqrt(0.25 * two_I * (two_I + 2) - M[1:] * (M[1:] + 1)), 1)
    return [0.5 * (up + up.T), -0.5j * (up - up.T), np.diag(M)]


class _Exact:
    """H - iK of one pair on states of shape (rows, d_last, ..., d_first, 2, 2): nuclei sorted by
    spin (stable), the first one next to the electrons (the layout the C header states)."""

    def __init__(self, s):
        self.s, self.dev = s, torch.device("cuda")
        self.order = [int(k) for k in np.argsort(s.two_I, kind="stable")]
        self.d = [int(s.two_I[k]) + 1 for k in self.order]
        self.Z = int(np.prod(self.d)) if self.d else 1
        S = _spin(1)
        dot = sum(np.kron(S[a], S[a]) for a in range(3))
        self.sz = torch.tensor(np.real(np.diag(np.kron(S[2], np.eye(2)) + np.kron(np.eye(2), S[2]))),
                               device=self.dev)
        E = (2.0 * GAMMA_E * s.J * dot - 0.5j * s.k_S * (0.25 * np.eye(4) - dot)
             - 0.5j * s.k_T * (0.75 * np.eye(4) + dot))
        self.E = torch.tensor(E, device=self.dev).T.contiguous()
        self.blocks, self.width, lo = [], abs(2.0 * GAMMA_E * s.J), 1
        for k, d in zip(self.order, self.d):
            I = _spin(d - 1)
            h = GAMMA_E * sum(s.A[k][a, b] * np.kron(S[a], I[b]) for a in range(3) for b in range(3))
            e = np.linalg.eigvalsh(h)
            self.width += 0.5 * (e[-1] - e[0])
            self.width += abs(0.5 * (e[-1] + e[0]))
            h = h.reshape(2, d, 2, d)
            nz = [(a, i, b, j, complex(h[a, i, b, j])) for a in range(2) for i in range(d)
                  for b in range(2) for j in range(d) if h[a, i, b, j] != 0]
            self.blocks.append((int(s.radical[k]), lo, d, nz))
            lo *= d
        self.csr = self._csr() if self.Z <= 32768 else None

    def _csr(self):
        """All of H - iK but the Zeeman term as one sparse 4Z x 4Z matrix."""
        Z, m = self.Z, torch.arange(self.Z, device=self.dev)
        rows, cols, vals = [], [], []

        def put(r, q, v):
            rows.append(r), cols.append(q)
            vals.append(torch.full((r.numel(),), v, dtype=torch.complex128, device=self.dev))
        E = self.E.T.cpu().numpy()
        for a in range(4):
            for b in range(4):
                if E[a, b] != 0:
                    put(4 * m + a, 4 * m + b, complex(E[a, b]))
        for r, lo, d, nz in self.blocks:
            dig = (m // lo) % d
            for a, i, b, j, v in nz:
                mi = m[dig == i]
                for o in range(2):
                    ea, eb = (2 * a + o, 2 * b + o) if r == 0 else (2 * o + a, 2 * o + b)
                    put(4 * mi + ea, 4 * (mi + (j - i) * lo) + eb, v)
        idx = torch.stack([torch.cat(rows), torch.cat(cols)])
        return torch.sparse_coo_tensor(idx, torch.cat(vals), (4 * Z, 4 * Z)).coalesce().to_sparse_csr()

    def apply(self, psi, omega):
        """(H - iK) psi for psi (rows, 4Z) complex128 and Zeeman omega (rows)."""
        R = psi.shape[0]
        v = psi.view(R, self.Z, 4)
        y = v * (omega[:, None, None] * self.sz[None, None, :])
        if self.csr is not None:
            return (y.view(R, -1) + (self.csr @ psi.T.contiguous()).T).contiguous()
        y += v @ self.E
        for r, lo, d, nz in self.blocks:
            a6, p6 = (t.view(R, self.Z // (lo * d), d, lo, 2, 2) for t in (y, v))
            for a, i, b, j, h in nz:
                if r == 0:
                    a6[:, :, i, :, a, :].add_(p6[:, :, j, :, b, :], alpha=h)
                else:
                    a6[:, :, i, :, :, a].add_(p6[:, :, j, :, :, b], alpha=h)
        return y.view(R, -1)

    def initial(self, seed, pair, samples, n_fields, basis):
        n = len(self.s.two_I)
        if basis is not None:
            nuc = np.zeros((len(basis), self.Z), complex)
            nuc[np.arange(len(basis)), basis] = 1.0
        else:
            u1, u2 = _philox(seed, pair, samples, n) if n else (None, None)
            nuc = np.ones((len(samples), 1), complex)
            for k, d in zip(self.order, self.d):
                j = np.arange(d)
                amp = (np.sqrt([math.comb(d - 1, q) for q in j]) * np.sqrt(1.0 - u1[:, k])[:, None] ** (d - 1 - j)
                       * np.sqrt(u1[:, k])[:, None] ** j * np.exp(2j * np.pi * u2[:, k][:, None] * j))
                nuc = (amp[:, :, None] * nuc[:, None, :]).reshape(len(samples), -1)
        sing = np.array([0.0, 1.0, -1.0, 0.0]) / math.sqrt(2.0)
        psi = torch.tensor(nuc, device=self.dev)[:, :, None] * torch.tensor(sing, device=self.dev)
        return psi.reshape(psi.shape[0], -1).repeat(n_fields, 1).contiguous()

    def propagate(self, psi, omega, h, n_steps, on_step=None):
        """n_steps of length h; returns psi and int |<S|psi>|^2 dt per row.  Each step is cut into
        parts of dE tau <= 30, a Chebyshev series of 80 terms and 48 Gauss-Legendre nodes."""
        dE = float(omega.abs().max()) + self.width + 1e-6
        parts = max(1, math.ceil(dE * h / 30.0))
        tau, n_c, q = h / parts, 80, 48
        gx, gw = np.polynomial.legendre.leggauss(q)
        tt = np.append(0.5 * tau * (gx + 1.0), tau)
        th = 2.0 * np.pi * np.arange(512) / 512
        Jn = np.real(np.fft.fft(np.exp(1j * dE * tt[:, None] * np.sin(th)), axis=1) / 512)[:, :n_c]
        co = torch.tensor(Jn * (2.0 - (np.arange(n_c) == 0)) * (-1j) ** (np.arange(n_c) % 4), device=self.dev)
        gw = torch.tensor(0.5 * tau * gw, device=self.dev)
        R, integral = psi.shape[0], torch.zeros(psi.shape[0], dtype=torch.float64, device=self.dev)
        S = torch.empty((n_c, R * self.Z), dtype=torch.complex128, device=self.dev)
        for step in range(n_steps):
            for _ in range(parts):
                p0, p1 = None, psi
                acc = co[q, 0] * psi
                for n in range(n_c):
                    if n == 1:
                        p0, p1 = p1, self.apply(p1, omega) / dE
                    elif n > 1:
                        p0, p1 = p1, self.apply(p1, omega) * (2.0 / dE) - p0
                    if n:
                        acc += co[q, n] * p1
                    v = p1.view(R, self.Z, 4)
                    S[n] = ((v[:, :, 1] - v[:, :, 2]) / math.sqrt(2.0)).reshape(-1)
                for i in range(0, q, 8):
                    x = (co[i:i + 8] @ S).view(-1, R, self.Z)
                    integral += (gw[i:i + 8, None] * (x.real ** 2 + x.imag ** 2).sum(dim=2)).sum(dim=0)
                psi = acc
            if on_step:
                on_step(step, psi)
        return psi, integral


def _groups(Z, M, n_fields):
    return 1 if Z * M * n_fields <= 1 << 20 else min(8, n_fields)


def _seconds(c, two_I, n_fields, T):
    """Rough time of _yields_exact (dE tau = 30 per 80 terms there, 46 or 56 per 88 in _terms)."""
    Z, n = float(np.prod(np.array(two_I) + 1.0)), max(len(two_I), 1)
    groups = _groups(Z, c["M"], n_fields)
    rows = c["M"] * n_fields / groups
    per = 1.2e-4 + rows * Z * 4 * 16 * 12 / 2e12 if Z <= 32768 else n * 3e-4 + rows * Z * 4 * 16 * 14 * n / 3e12
    return per * 2.0 * _terms(c, two_I, c["B_max"], T) * (groups if groups == 1 else 0.55 * groups)


def _yields_exact(s, c, fields, T, seed, pair, basis=None):
    ex = _Exact(s)
    M = len(basis) if basis is not None else c["M"]
    omega = torch.tensor(np.repeat(GAMMA_E * fields, M), device="cuda")
    psi = ex.initial(seed, pair, np.arange(M), len(fields), basis)
    # groups of rows whose field is alike (a small field needs fewer parts) where the work counts
    surv, integral = torch.empty_like(omega), torch.empty_like(omega)
    order = torch.argsort(omega)
    for rows in torch.chunk(order, _groups(ex.Z, M, len(fields))):
        p, i = ex.propagate(psi[rows].contiguous(), omega[rows], T, 1)
        integral[rows] = i
        surv[rows] = (p.real ** 2 + p.imag ** 2).sum(dim=1)
    phi = s.k_S * integral.cpu().numpy().reshape(len(fields), M)
    surv = surv.cpu().numpy().reshape(len(fields), M)
    ps = np.stack([phi, 1.0 - surv - phi, surv], axis=2)
    m, se = ps.mean(axis=1), ps.std(axis=1, ddof=1) / math.sqrt(M)
    return np.stack([m[:, 0], m[:, 1], se[:, 0], se[:, 1], m[:, 2]], axis=1), ps


def _trace_steps(c, s):
    """Macro-steps of the time grid for k_S = k_T: dE h as large as the tail of the Chebyshev series,
    2 sum_{n >= n_cheb} |J_n(dE h)|, stays below the tolerance; dE from the sum of the blocks' spectra."""
    w, Je = GAMMA_E * c["B_max"], GAMMA_E * c["J"]
    ev = [w + 0.5 * Je, 0.5 * Je, -w + 0.5 * Je, -1.5 * Je]
    dE = 0.5 * (max(ev) - min(ev))
    for k, t in enumerate(s.two_I):
        I, S = _spin(int(t)), _spin(1)
        e = np.linalg.eigvalsh(GAMMA_E * sum(s.A[k][a, b] * np.kron(S[a], I[b]) for a in range(3) for b in range(3)))
        dE += 0.5 * (e[-1] - e[0])
    lo, hi = 1.0, float(N_CHEB)
    for _ in range(50):
        x = 0.5 * (lo + hi)
        J = [0.0] * 250 + [1e-250, 0.0]  # downward recurrence, normalised by J_0 + 2 sum J_2k = 1
        for n in range(250, 0, -1):
            J[n - 1] = 2.0 * n / x * J[n] - J[n + 1]
        tail = 2.0 * sum(abs(v) for v in J[N_CHEB:208]) / abs(2.0 * sum(J[0::2]) - J[0])
        lo, hi = (x, hi) if tail <= (1e-15 if c["precision"] == "fp64" else 1e-9) else (lo, x)
    return math.ceil(dE * c["T"] / lo)


def exact(case, seed):
    c = dict(case)
    pairs, fields = _inputs(c, seed), _fields(c)
    if c["kind"] == "cv":
        return _cv_exact(c, pairs[0][0], fields, seed)
    s, T = pairs[0]
    if c["kind"] == "apply":
        ex = _Exact(s)
        x = torch.tensor(_apply_vectors(c, ex.Z, seed).astype(np.float64), device="cuda")
        om = torch.full((c["M"],), GAMMA_E * c["B_max"], dtype=torch.float64, device="cuda")
        y = torch.view_as_real(ex.apply(torch.view_as_complex(x), om))
        return {"y": y.reshape(x.shape)}
    cost = sum(_seconds(c, [int(v) for v in sp.two_I], len(fields), Tp) for sp, Tp in pairs)
    if cost > 7.5 or c["deterministic"]:
        return None
    if c["kind"] == "batch":
        return {"out": np.stack([_yields_exact(sp, c, fields, Tp, seed, i)[0]
                                 for i, (sp, Tp) in enumerate(pairs)])}
    if c["kind"] == "yields":
        out, ps = _yields_exact(s, c, fields, T, seed, 0)
        return {"out": out, "per_sample": ps}
    if c["k_S"] != c["k_T"]:
        return None
    ex, n = _Exact(s), _trace_steps(c, s)
    psi = ex.initial(seed, 0, np.arange(c["M"]), 1, None)
    om = torch.full((c["M"],), GAMMA_E * c["B_max"], dtype=torch.float64, device="cuda")
    out = np.zeros((n + 1, 3))
    out[0] = 1.0, 0.0, 1.0

    def at(step, p):
        v = p.view(c["M"], ex.Z, 4)
        ps = float((0.5 * (v[:, :, 1] - v[:, :, 2]).abs() ** 2).sum()) / c["M"]
        nn = float((v.abs() ** 2).sum()) / c["M"]
        out[step + 1] = ps, nn - ps, nn
    ex.propagate(psi, om, T / n, n, at)
    return {"t": np.arange(n + 1) * (T / n), "out": out}


def _cv_exact(c, s, fields, seed):
    n = len(s.two_I)
    p, dims = _cv_params(c, 3 * n + 10, seed)
    net, o = [], 0
    for a, b in zip(dims[:-1], dims[1:]):
        W = torch.from_numpy(p[o:o + a * b]).reshape(b, a).cuda().bfloat16().double()
        net.append((W, torch.from_numpy(p[o + a * b:o + a * b + b]).cuda().double()))
        o += a * b + b
    I = 0.5 * np.asarray(s.two_I)
    bh = [math.sqrt(sum((s.A[k] ** 2).sum() / 3.0 * I[k] * (I[k] + 1) for k in range(n) if s.radical[k] == r))
          for r in (0, 1)]

    def g_of(samples, B):
        u1, u2 = _philox(seed, 0, samples, n)
        ct = 1.0 - 2.0 * u1
        st = np.sqrt(np.maximum(0.0, 1.0 - ct * ct))
        v = np.stack([st * np.cos(2 * np.pi * u2), st * np.sin(2 * np.pi * u2), ct], axis=2)
        b = [sum((v[:, k] @ (I[k] * s.A[k] / bh[r]).T for k in range(n) if s.radical[k] == r),
                 np.zeros((len(samples), 3))) for r in (0, 1)]
        x = np.concatenate([v.reshape(len(samples), -1), b[0], b[1], np.linalg.norm(b[0], axis=1)[:, None],
                            np.linalg.norm(b[1], axis=1)[:, None], (b[0] * b[1]).sum(axis=1)[:, None],
                            np.broadcast_to(np.asarray(B) / 10.0, (len(samples),))[:, None]], axis=1)
        h = torch.from_numpy(x).cuda()
        for l, (W, bias) in enumerate(net):
            h = h @ W.T + bias
            if l + 1 < len(net):
                h = h * torch.sigmoid(h)
        return h[:, 0]
    mu, vm = [], []
    for B in fields:
        g = torch.cat([g_of(np.arange(i, min(i + 16384, c["n_mc"])), B) for i in range(0, c["n_mc"], 16384)])
        mu.append(float(g.mean()))
        vm.append(float(g.var()) / c["n_mc"])
    g = g_of(np.arange(c["M"]), np.resize(fields, c["M"]))
    return {"mu": np.array(mu), "var_mu": np.array(vm), "g": g}
