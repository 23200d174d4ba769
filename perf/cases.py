"""Workloads of the density-matrix RT-TDDFT library, as its users run them.

A case is one context (one or several synthetic systems, a propagator, a
precision mode, truncation radii) and one pass over it:

  * "run": set the density (or restore a checkpoint, CN), advance `steps` time
    steps, read the observables of every (system, kick) pair and the updated
    density matrices back;
  * "setup": the set-up a new geometry pays for -- Hotelling S^-1, the
    Chebyshev ground state, the delta kick -- and the density read back.

Sizes are the repository's own (diamond cells of 64 to 1728 atoms with 4 and 13
functions, the H-terminated Si cluster; radii 6 to 10 A; x, y and z kicks).
"""
import dataclasses
import functools
import math

import numpy as np
import torch

import paper_1404_5776_gb300 as rt
import synth

KAPPA = 1e-3          # delta kick (a.u.)
DT = 0.05             # time step (a.u.)
DENSE_K0 = 900        # up to this many functions K0 is a dense diagonalisation, above it the library's Chebyshev
                      # expansion
FOE_ORDER, FOE_KT = 30, 0.02
# chemical potential (mid-gap) and spectral bounds of S^-1 H0 of the two diamond models, with the margin of 0.5 Ha
# that the benchmark takes
SPECTRUM = {"sp4": (-0.33, -1.25, 1.0), "spd13": (-0.395, -1.75, 2.1)}
PULSE = dict(E0=5e-3, t0=0.5, sigma=0.3, omega=0.6)  # Gaussian pulse of the propagator study


def _case(name, systems, steps, radius, **kw):
    c = dict(name=name, kind="run", systems=systems, steps=steps, r_SH=7.0 if "spd13" in systems else 6.0,
             r_Sinv=radius, r_T=radius, r_U=radius, r_K=radius, r_M=radius, prop="em", precision="fp64",
             full_step=1, field_poly=0, incremental=0, n_kick=1, pulse=False)
    c.update(kw)
    return c


def listed():
    split = dict(precision="fp32", incremental=1)
    return [
        # the smallest calls: a 64-atom 4-function cell, FP64 EM (the golden-trajectory workload); bound by launches
        _case("fp64_em_64x4", "sp4:2", 20, 8.0),
        # the library's default mode (FP64, EM full step) on 13-function atoms under a Gaussian pulse
        _case("fp64_em_216x13_pulse", "spd13:3", 4, 8.0, pulse=True),
        # the same at the largest FP64 size here: the "plain FP64 path" that every mixed result is compared with
        _case("fp64_em_512x13", "spd13:4", 2, 8.0),
        # 4-function atoms in FP64: the linear-scaling systems without mixed precision
        _case("fp64_em_1728x4", "sp4:6", 4, 8.0),
        # Crank-Nicolson with the warm-started Hotelling inverse, resumed from a checkpoint
        _case("fp64_cn_64x13", "spd13:2", 3, 8.0, prop="cn"),
        # the mixed reference split (the benchmark's path), small: one cell, spectra of small systems
        _case("split_em_64x13", "spd13:2", 50, 8.0, full_step=1, field_poly=1, **split),
        # the same at an ordinary size, field polynomial every step
        _case("split_em_512x13", "spd13:4", 60, 8.0, full_step=1, field_poly=1, **split),
        # the benchmark's radius, 10 A, after a delta kick: U built once, propagation steps
        _case("split_const_216x13_r10", "spd13:3", 30, 10.0, full_step=0, **split),
        # the literal mixed path under a pulse: Taylor powers and sandwich as FP32 products
        _case("mixed_em_216x13_pulse", "spd13:3", 8, 8.0, precision="fp32", pulse=True),
        # x, y and z kicks of systems of uneven size and block size (13, 1+4, 4 functions) in one context
        _case("split_batch_3kicks", "spd13:2,si_h:60,sp4:3", 20, 6.5, n_kick=3, full_step=1, field_poly=1, **split),
        # the linear-scaling sweep's step: 4-function atoms, three kicks
        _case("split_em_1728x4_3kicks", "sp4:6", 20, 8.0, n_kick=3, full_step=1, field_poly=1, **split),
        # what a new geometry costs before the first step
        _case("setup_216x13", "spd13:3", 0, 8.0, kind="setup"),
    ]


def draw(rng):
    """One more case of the same ranges; radii differ between the matrices, and sizes between the systems."""
    most = max(_cost(c) for c in listed())
    while True:
        radius = lambda: round(rng.uniform(5.0, 8.5 if rng.random() < 0.7 else 10.0), 2)
        path = rng.choice(["fp64", "fp64", "split", "split", "split_const", "mixed", "setup"])
        n_sys = rng.choice([1, 1, 2, 3]) if path != "setup" else 1
        names = []
        for _ in range(n_sys):
            basis = rng.choice(["sp4", "spd13", "spd13"] + (["si_h"] if path != "setup" else []))
            names.append("si_h:%d" % rng.choice([30, 60, 90, 150]) if basis == "si_h" else
                         "%s:%d" % (basis, rng.choice([2, 2, 3, 4] if basis == "spd13" and n_sys == 1 else [2, 3] if basis == "spd13" else
                                         [2, 3, 4, 5, 6] if n_sys == 1 else [2, 3, 4])))
        systems = ",".join(names)
        r_K = radius()
        c = _case("", systems, max(1, int(math.exp(rng.uniform(0.0, math.log(60.0))))), r_K, r_U=radius(),
                  r_M=round(r_K + rng.choice([0.0, 0.0, 0.75]), 2), r_Sinv=round(rng.uniform(6.5, 9.0), 2),
                  r_T=round(rng.uniform(6.5, 9.0), 2), n_kick=rng.choice([1, 1, 2, 3]), pulse=rng.random() < 0.4)
        if rng.random() < 0.5:  # one radius for the step's matrices, as the benchmark has it
            c.update(r_U=r_K, r_M=r_K)
        if path == "fp64":
            c["prop"] = rng.choice(["em", "em", "etrs", "m4", "cn"])
            c["field_poly"] = int(c["prop"] == "em" and rng.random() < 0.3)
        elif path == "split":
            c.update(precision="fp32", incremental=1, field_poly=1)
        elif path == "split_const":
            c.update(precision="fp32", incremental=1, full_step=0, pulse=False, prop=rng.choice(["em", "em", "cn"]))
        elif path == "mixed":
            c.update(precision="fp32", prop=rng.choice(["em", "em", "etrs", "m4"]))
        else:
            c.update(kind="setup", steps=0, n_kick=1, pulse=False, systems=systems.replace("spd13:4", "spd13:3"))
        del c["name"]
        while c["steps"] > 1 and _cost(c) > most:
            c["steps"] //= 2
        if _cost(c) <= most:
            return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
@functools.lru_cache(maxsize=None)
def _geometry(item, r, k):
    """One system of the synthetic model, and where the diagonals of its on-site blocks of H0 lie."""
    kind, n = item.split(":")
    if kind == "si_h":
        pos, species = synth.si_h_cluster(target=int(n))
        pos = pos + 0.02 * np.random.default_rng(k).normal(size=pos.shape)
        s = synth.build_system(pos, None, species, r, r)
    else:
        s = synth.diamond_system(int(n), kind, r, r, seed=k)
    off = s.block_offsets(s.h_rowptr, s.h_col)
    rows = np.repeat(np.arange(s.n_atoms), np.diff(s.h_rowptr))
    on_site = off[:-1][rows == s.h_col]
    return s, np.concatenate([o + (b + 1) * np.arange(b) for o, b in zip(on_site, s.bsize)])


def _systems(case, seed):
    """The geometry, and so every pattern, is the case's; the on-site energies of H0 are the seed's (another K0, another
    response), as in a run over disorder samples."""
    out = []
    for k, item in enumerate(case["systems"].split(",")):
        s, diagonal = _geometry(item, case["r_SH"], k)
        h = s.h_val.copy()
        h[diagonal] += np.random.default_rng([seed, k]).uniform(-0.05, 0.05, size=len(diagonal))
        out.append(dataclasses.replace(s, h_val=h))
    return out


def _basis(case, k):
    return case["systems"].split(",")[k].split(":")[0]


def _params(case):
    names = ("r_Sinv", "r_T", "r_U", "r_K", "r_M", "prop", "precision", "full_step", "field_poly", "incremental",
             "n_kick")
    return dict({n: case[n] for n in names}, dt=DT)


def _field(case):
    return dict(kind=rt.RT_FIELD_GAUSSIAN, dir=0, **PULSE) if case["pulse"] else dict(kind=rt.RT_FIELD_NONE)


def _dense_k0(s):
    return synth.ground_state_dense(s, int(np.sum(s.bsize)) // 2 if len(set(s.bsize)) > 1 else 2 * s.n_atoms)[0]


class State:
    pass


def prepare(case, seed):
    """The context with its inverse formed and K(0+) in pinned host memory (or a checkpoint, CN)."""
    st = State()
    st.case = case
    st.systems = _systems(case, seed)
    st.ctx = rt.RT(st.systems, **_params(case))
    st.ctx.set_field(**_field(case))
    if case["kind"] == "setup":
        return st
    ctx = st.ctx
    ctx.inverse()
    st.k0 = []
    for si, s in enumerate(st.systems):
        if s.n > DENSE_K0:
            mu, lo, hi = SPECTRUM[_basis(case, si)]
            ctx.ground_state(si, FOE_ORDER, mu, FOE_KT, lo, hi)
        for k in range(case["n_kick"]):
            if s.n <= DENSE_K0:
                dense = _dense_k0(s) if k == 0 else dense
                ctx.set_density_dense(si, k, dense)
            if not case["pulse"]:
                ctx.kick(si, k, k, KAPPA)
    for si in range(len(st.systems)):
        for k in range(case["n_kick"]):
            host = torch.from_numpy(ctx.matrix(si, rt.RT_MAT_K, k))
            st.k0.append((si, k, host.pin_memory() if torch.cuda.is_available() else host))
    if not case["full_step"]:
        ctx.propagator(0.0)
    st.checkpoint = ctx.get_state() if case["prop"] == "cn" and case["full_step"] else None
    return st


def run(st):
    ctx, case = st.ctx, st.case
    if case["kind"] == "setup":
        ctx.inverse()
        mu, lo, hi = SPECTRUM[_basis(case, 0)]
        ctx.ground_state(0, FOE_ORDER, mu, FOE_KT, lo, hi)
        ctx.kick(0, 0, 0, KAPPA)
        return [ctx.matrix(0, rt.RT_MAT_SINV), ctx.matrix(0, rt.RT_MAT_K)]
    if st.checkpoint is not None:
        ctx.set_state(st.checkpoint)
    else:
        for si, k, host in st.k0:
            ctx.set_density(si, k, host.numpy())
    ctx.step(case["steps"])
    out = []
    for si, k, _ in st.k0:
        out.append(ctx.observables(si, k, case["steps"]))
        out.append(ctx.matrix(si, rt.RT_MAT_K, k))
    return out


# ---------------------------------------------------------------------------
# work
# ---------------------------------------------------------------------------
_counts, _sites = {}, {}


def _within(a, b, cell, r):
    """Whether each atom of `b` is within r of each of `a` (minimum image), by the pattern rule of the library."""
    d = b[None, :, :] - a[:, None, :]
    if cell is not None:
        d -= cell * np.rint(d / cell)
    return (d[..., 0] * d[..., 0] + d[..., 1] * d[..., 1]) + d[..., 2] * d[..., 2] < r * r


def _triples(item, ra, rb, rc):
    """Block triples (i,k,j) of a product cut to rc, and the blocks of P_rc, from some of the rows in larger systems."""
    if item not in _sites:
        kind, n = item.split(":")
        _sites[item] = (synth.si_h_cluster(target=int(n))[0], None) if kind == "si_h" else synth.diamond_positions(int(n))
    key = (item, ra, rb, rc)
    if key not in _counts:
        pos, cell = _sites[item]
        n = len(pos)
        rows = np.arange(n) if n <= 64 else np.linspace(0, n - 1, 16).astype(int)
        triples = blocks = 0
        for i in rows:
            a, c = (pos[_within(pos[i:i + 1], pos, cell, r)[0]] for r in (ra, rc))
            triples += int(_within(a, c, cell, rb).sum())
            blocks += len(c)
        _counts[key] = triples * n / len(rows), blocks * n / len(rows)
    return _counts[key]


def _flops_bytes(case):
    """Multiply-adds of the products of one pass (true block sizes; the cluster's mix of 1 and 4 functions as 2.7) and
    the values that it has to read and write: the given matrices and K in, K and the observables out."""
    flops = total = 0.0
    c = case
    rs = c["r_SH"]
    for item in c["systems"].split(","):
        b = {"sp4": 4.0, "spd13": 13.0, "si_h": 2.7}[item.split(":")[0]]
        real, cplx = 2.0 * b ** 3, 8.0 * b ** 3
        tri = lambda *r: _triples(item, *r)[0]
        T = tri(c["r_Sinv"], rs, c["r_T"])
        taylor = tri(c["r_T"], c["r_T"], c["r_U"]) + 3.0 * tri(c["r_T"], c["r_U"], c["r_U"])
        sandwich = tri(c["r_U"], c["r_K"], c["r_M"]) + 0.5 * tri(c["r_M"], c["r_U"], c["r_K"])
        nK = _triples(item, c["r_K"], rs, c["r_K"])[1]
        nS = _triples(item, rs, rs, rs)[1]
        total += b * b * (8.0 * 5.0 * nS)
        if c["kind"] == "setup":
            # about 12 Hotelling iterations of two products, the Chebyshev terms, T and the kick's Taylor series
            hot = 12.0 * (tri(rs, c["r_Sinv"], c["r_Sinv"]) + tri(c["r_Sinv"], c["r_Sinv"], c["r_Sinv"]))
            foe = FOE_ORDER * tri(c["r_T"], c["r_K"], c["r_K"])
            flops += real * (hot + foe + 2.0 * T + taylor + 7.0 * tri(c["r_T"], c["r_U"], c["r_U"])) + cplx * sandwich
            total += b * b * 24.0 * nK
            continue
        if c["prop"] == "cn":
            ab = 2.0 * (tri(rs, c["r_U"], c["r_U"]) + tri(c["r_U"], c["r_U"], c["r_U"])) + tri(c["r_U"], rs, c["r_U"])
            build = cplx * ab
        elif c["prop"] == "etrs":
            build = 2.0 * real * (T + taylor) + cplx * tri(c["r_U"], c["r_U"], c["r_U"])
        elif c["prop"] == "m4":
            build = real * 2.0 * (T + tri(c["r_T"], c["r_T"], c["r_U"])) + cplx * 4.0 * tri(c["r_U"], c["r_U"], c["r_U"])
        else:
            build = real * (T + taylor)
        if not c["full_step"] or c["field_poly"]:
            build = 0.0
        flops += c["steps"] * (build + cplx * c["n_kick"] * sandwich)
        total += b * b * 32.0 * nK * c["n_kick"]
    return flops, total


def _cost(case):
    """Estimated seconds: FP64 products at 1.1 TFLOP/s, FP32 ones at 25, and a few ms a GB for the host copies."""
    flops, total = _flops_bytes(case)
    return flops / (1.1e12 if case["precision"] == "fp64" else 25e12) + total / 1e9


def work(case):
    flops, total = _flops_bytes(case)
    return {"bytes": total, "flops": flops}


# ---------------------------------------------------------------------------
# the same in plain dense 64-bit algebra
# ---------------------------------------------------------------------------
class _Dense:
    """One system's matrices as dense n x n tensors, and the cut of each radius as a mask."""

    def __init__(self, s, case):
        self.dev = "cuda" if torch.cuda.is_available() else "cpu"
        self.s, self.case = s, case
        to = lambda a: torch.as_tensor(a, dtype=torch.float64, device=self.dev)
        self.S, self.H = to(s.to_dense("S")), to(s.to_dense("H"))
        self.D = [to(s.to_dense(w)) for w in ("Dx", "Dy", "Dz")]
        self.atom = torch.as_tensor(np.repeat(np.arange(s.n_atoms), s.bsize), device=self.dev)
        self.masks = {}

    def cut(self, M, r):
        if r not in self.masks:
            m = torch.as_tensor(_within(self.s.pos, self.s.pos, self.s.cell, r), device=self.dev)
            self.masks[r] = m[self.atom][:, self.atom]
        return M * self.masks[r]

    def inverse(self, tol=1e-10):
        r, n = self.case["r_Sinv"], self.s.n
        eye = torch.eye(n, dtype=torch.float64, device=self.dev)
        X, prev = eye / self.S.abs().sum(1).max(), None
        for it in range(101):
            Z = 2.0 * eye - self.cut(self.S @ X, r)
            res = float(torch.linalg.norm(Z - eye)) / math.sqrt(n)
            if res < tol or (prev is not None and res > 0.9 * prev):
                break
            X, prev = self.cut(X @ Z, r), res
        self.X, self.eye = X, eye
        return X

    def ground_state(self, mu, lo, hi):
        r, N = self.case["r_K"], FOE_ORDER
        T = self.cut(self.X @ self.H, self.case["r_T"])
        a, w = 0.5 * (hi + lo), 0.5 * (hi - lo)
        th = math.pi * (np.arange(4 * (N + 1)) + 0.5) / (4 * (N + 1))
        f = 0.5 * (1.0 - np.tanh(0.5 * (a + w * np.cos(th) - mu) / FOE_KT))
        coef = [(2.0 if n else 1.0) / len(th) * float(np.sum(f * np.cos(n * th))) for n in range(N + 1)]
        Y = self.cut(self.X, r)
        K, Yp = coef[0] * Y, None
        for n in range(1, N + 1):
            XY = (self.cut(T @ Y, r) - a * Y) / w
            Y, Yp = (XY, Y) if Yp is None else (2.0 * XY - Yp, Y)
            K = K + coef[n] * Y
        return (0.5 * (K + K.T)).to(torch.complex128)

    def series(self, T, dt, terms, r):
        """sum_{n < terms} (-i dt)^n T^n / n!, the powers cut to r."""
        U, P, c = torch.complex(self.eye, -dt * self.cut(T, r)), T, -1j * dt
        for n in range(2, terms):
            P = self.cut(T @ P, r)
            c = c * (-1j * dt) / n
            U = U + c * P
        return U

    def sandwich(self, U, K):
        M = self.cut(U @ K, self.case["r_M"])
        N = self.cut(M @ U.conj().T, self.case["r_K"])
        i, j = self.atom[:, None], self.atom[None, :]
        up, on = (j > i).to(N.real.dtype), (j == i).to(N.real.dtype)
        return N * up + (N * up).conj().T + 0.5 * (N + N.conj().T) * on

    def kick(self, K, d):
        T = self.cut(self.X @ self.D[d], self.case["r_T"])
        return self.sandwich(self.series(T, -KAPPA, 12, self.case["r_U"]), K)

    def propagator(self, t):
        c, dt, rU, rT = self.case, DT, self.case["r_U"], self.case["r_T"]

        def T(at):
            return self.cut(self.X @ self.hamiltonian(at), rT)

        if c["prop"] == "em":
            return self.series(T(t + 0.5 * dt), dt, 6, rU)
        if c["prop"] == "etrs":
            return self.cut(self.series(T(t + dt), 0.5 * dt, 6, rU) @ self.series(T(t), 0.5 * dt, 6, rU), rU)
        if c["prop"] == "m4":
            T1, T2 = T(t + (0.5 - math.sqrt(3) / 6) * dt), T(t + (0.5 + math.sqrt(3) / 6) * dt)
            om = torch.complex(-math.sqrt(3) * dt * dt / 12 * (self.cut(T2 @ T1, rU) - self.cut(T1 @ T2, rU)),
                               -0.5 * dt * self.cut(T1 + T2, rU))
            U, P, f = self.eye + om, om, 1.0
            for n in range(2, 6):
                P, f = self.cut(om @ P, rU), f / n
                U = U + f * P
            return U
        H = self.hamiltonian(t + 0.5 * dt)
        A, B = torch.complex(self.S, 0.5 * dt * H), torch.complex(self.S, -0.5 * dt * H)
        if self.warm is None:
            self.warm = self.cut(self.X, rU).to(torch.complex128)
        for _ in range(2):
            Y = self.cut(A @ self.warm, rU)
            self.resid = float(torch.linalg.norm(self.cut(self.eye, rU) - Y)) / math.sqrt(self.s.n)
            self.warm = self.cut(self.warm @ (2.0 * self.eye - Y), rU)
        return self.cut(self.warm @ B, rU)

    def hamiltonian(self, t):
        if not self.case["pulse"]:
            return self.H
        x = t - PULSE["t0"]
        return self.H - PULSE["E0"] * math.exp(-x * x / (2.0 * PULSE["sigma"] ** 2)) * math.cos(PULSE["omega"] * x) * self.D[0]

    def blocks(self, M, r):
        """The values of the kept blocks, row-major, in pattern order."""
        s = self.s
        m = _within(s.pos, s.pos, s.cell, r)
        off = np.concatenate([[0], np.cumsum(s.bsize)])
        M = M.to(torch.complex128).cpu().numpy()
        return np.concatenate([M[off[i]:off[i + 1], off[j]:off[j + 1]].reshape(-1) for i in range(s.n_atoms)
                               for j in np.nonzero(m[i])[0]])

    def run(self, K, steps):
        obs, t = np.zeros((steps, rt.RT_NOBS)), 0.0
        self.warm = self.resid = None
        U = None
        traced = [self.S] + self.D
        for n in range(steps):
            if U is None or self.case["pulse"] or self.case["prop"] == "cn":  # a constant H has a constant U
                if self.case["full_step"] or U is None:
                    U = self.propagator(t)
            K = self.sandwich(U, K)
            t += DT
            obs[n, 0] = t
            for k, X in enumerate(traced):
                obs[n, 1 + 2 * k] = float((K.real * X.T).sum())  # the imaginary parts of a hermitian K's traces are 0
            if self.case["prop"] == "cn" and self.case["full_step"]:
                obs[n, 10], obs[n, 11] = 2, self.resid
        return [obs, self.blocks(K, self.case["r_K"])]


def exact(case, seed):
    systems = _systems(case, seed)
    n3 = sum(float(s.n) ** 3 for s in systems)
    if case["kind"] == "setup":
        flops = n3 * 2 * (FOE_ORDER + 40)
    else:
        moving = case["pulse"] or (case["prop"] == "cn" and case["full_step"])
        flops = n3 * (140 + (FOE_ORDER * 2 if n3 > DENSE_K0 ** 3 else 0) + (60 if moving else 0) * case["steps"]
                      + 16 * case["steps"] * case["n_kick"])
    if flops > 1.9e13 or max(s.n for s in systems) > 3500:
        return None  # minutes, or too large
    out = []
    for si, s in enumerate(systems):
        d = _Dense(s, case)
        d.inverse()
        if case["kind"] == "setup" or s.n > DENSE_K0:
            K0 = d.ground_state(*SPECTRUM[_basis(case, si)])
        else:
            K0 = d.cut(torch.as_tensor(_dense_k0(s), device=d.dev).to(torch.complex128), case["r_K"])
        if case["kind"] == "setup":
            return [d.blocks(d.X, case["r_Sinv"]), d.blocks(d.kick(K0, 0), case["r_K"])]
        for k in range(case["n_kick"]):
            out += d.run(K0 if case["pulse"] else d.kick(K0, k), case["steps"])
    return out
