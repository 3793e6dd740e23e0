"""The calls this framework is used for, with their inputs, work and 64-bit results.

A case is one call of a user's program on a system it holds a context for: some
time steps with the record read back, the operator on a block, the gradient of
the dipole, or the split-BF16 product on its own.  The systems have the shapes
of the configurations in synth/system.py (and their distributions), drawn on
the GPU from the seed; the trial vectors are the ground-state vectors that such
a program brings along, so that the context's Ritz step only confirms them.

Where a form keeps FP32 or split 16-bit accuracy, the results that carry it are
kept in 32 bits by the program; everything else stays in 64.  The record's
norm_dev and resid (the largest rounding error of a step) are not returned.
"""
import math

import numpy as np
import torch

from paper_2403_04351_gb300 import Context, rttddft

C_LIGHT = 137.035999084
BOHR = 1.0 / 0.529177210903
MOS2_A, MOS2_C = 3.16 * BOHR, 14.71 * BOHR
LATTICES = {
    "h2box": np.diag([21.401, 20.0, 20.0]),
    "mos2": np.array([[3 * MOS2_A, 0.0, 0.0], [1.5 * MOS2_A, 1.5 * MOS2_A * math.sqrt(3.0), 0.0], [0.0, 0.0, MOS2_C]]),
    "chain": np.diag([6.0, 6.0, 120.0]),
}

# shapes of the repository's configurations: cell, atoms, lmax, local orbitals
# per atom, states, auxiliary vectors (how many is a question of convergence,
# so the cases vary it), time step
TINY = dict(lattice="h2box", n_k=1, n_atoms=2, lmax=4, n_lo=20, n_s=8, n_aux=32, dt=0.1)
H2 = dict(lattice="h2box", n_k=1, n_atoms=2, lmax=8, n_lo=50, n_s=2, n_aux=200, dt=0.2)
CO = dict(lattice="h2box", n_k=1, n_atoms=2, lmax=8, n_lo=100, n_s=7, n_aux=400, dt=0.2)
MOS2 = dict(lattice="mos2", n_k=1, n_atoms=22, lmax=8, n_lo=5, n_s=60, n_aux=300, dt=0.2)


def step_case(base, n_g, precision, interstitial, steps, graph, drive="field", **kw):
    return dict(base, op="step", n_g=n_g, precision=precision, interstitial=interstitial, steps=steps, graph=graph,
                drive=drive, **kw)


def listed():
    return [
        # the smallest system with every option at its default (FP64, direct sum): launches and latency count
        dict(step_case(TINY, 360, "fp64", "toeplitz", 20, 10), name="tiny_fp64"),
        # the large-cell molecule as a first run does it: FP64, direct interstitial sum
        dict(step_case(H2, 5900, "fp64", "toeplitz", 10, 10), name="h2_fp64"),
        # the same system in its fast form, the long runs behind a spectrum
        dict(step_case(H2, 5900, "fp32", "fft", 20, 10), name="h2_fp32_fft"),
        # the potential rebuilt every step from the density it evolves
        dict(step_case(H2, 5900, "fp64", "fft", 4, 2, "hartree", mt_u=0.5), name="h2_fp64_hartree"),
        # gradient of the dipole with respect to the pulse (pulse design), checkpointed
        dict(H2, op="adjoint", n_g=5900, precision="fp64", interstitial="toeplitz", steps=60, ckpt=20, name="h2_adjoint"),
        # the second molecule in the tensor-core form
        dict(step_case(dict(CO, n_aux=240), 11800, "bf16x3", "fft", 10, 5), name="co_bf16x3_fft"),
        # its largest basis, in FP64 with the FFT route
        dict(step_case(dict(CO, n_aux=240), 25527, "fp64", "fft", 4, 2), name="co_large_fp64_fft"),
        # the operator alone on a block of vectors (checks, other propagators), more columns than states
        dict(CO, op="apply", n_aux=48, n_g=11800, precision="fp32", interstitial="toeplitz", n_cols=17, name="co_apply_fp32"),
        # the heterostructure, batched over k-points of unequal size, in the headline form
        dict(step_case(dict(MOS2, n_k=2), 7311, "bf16x3", "toeplitz", 5, 5), name="interface_bf16x3"),
        # one of its k-points in FP64, the reference form
        dict(step_case(dict(MOS2, n_aux=200), 7311, "fp64", "fft", 2, 2), name="interface_fp64_fft"),
        # a prescribed potential change rebuilt every step
        dict(step_case(dict(MOS2, n_atoms=14, n_aux=240), 6890, "bf16x3", "fft", 4, 2, "dv"), name="interface_bf16x3_fft_dv"),
        # the split-BF16 product alone: a tall basis block times a ragged set of states
        dict(op="zgemm", m=9917, n=61, k=300, trans=0, name="zgemm_bf16x3"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more call of the same kinds: sizes log-uniform between the listed ones, odd ones among them."""
    kind = rng.choice(["small", "molecule", "molecule", "interface", "interface", "dv", "hartree", "adjoint", "apply", "zgemm"])
    graph = rng.choice([1, 2, 5])
    if kind == "small":
        base = dict(TINY, n_s=rng.randint(1, 8), n_aux=rng.randint(16, 64), n_lo=rng.randint(5, 20))
        return step_case(base, _log(rng, 120, 900), rng.choice(["fp64", "fp32", "bf16x3", "fp16x3"]),
                         rng.choice(["toeplitz", "fft"]), 4 * graph, graph)
    if kind == "molecule":
        base = dict(rng.choice([H2, CO]), n_s=rng.randint(2, 9), n_aux=rng.randint(100, 240))
        route = rng.choice(["toeplitz", "fft"])
        return step_case(base, _log(rng, 2000, 12000 if route == "toeplitz" else 25000),
                         rng.choice(["fp64", "fp64", "fp32", "bf16x3", "fp16x3"]), route, 2 * graph, graph)
    if kind == "interface":
        prec = rng.choice(["fp64", "fp32", "bf16x3", "bf16x3", "fp16x3"])
        route = "fft" if prec in ("fp64", "fp32") else rng.choice(["toeplitz", "fft"])
        base = dict(MOS2, n_atoms=rng.randint(6, 22), n_s=rng.randint(12, 64), n_aux=rng.randint(100, 300))
        return step_case(base, _log(rng, 2500, 6500), prec, route, 2, 2)
    if kind == "dv":
        base = dict(MOS2, n_atoms=rng.randint(2, 12), n_s=rng.randint(4, 60), n_aux=rng.randint(100, 240))
        return step_case(base, _log(rng, 2500, 6500), rng.choice(["fp64", "fp32", "bf16x3"]), "fft", 2, 2, "dv")
    if kind == "hartree":
        base = dict(H2, n_s=rng.randint(2, 8), n_aux=rng.randint(60, 200), lattice=rng.choice(["h2box", "chain"]))
        return step_case(base, _log(rng, 600, 5900), rng.choice(["fp64", "fp32"]), "fft", 4, 2, "hartree", mt_u=rng.choice([0.0, 0.5]))
    if kind == "adjoint":
        return dict(H2, op="adjoint", n_g=_log(rng, 600, 5900), n_s=rng.randint(1, 12), n_aux=rng.randint(40, 240),
                    precision="fp64", interstitial="toeplitz", steps=rng.randint(15, 60), ckpt=rng.choice([7, 10, 50]))
    if kind == "apply":
        return dict(rng.choice([H2, CO]), op="apply", n_aux=rng.randint(24, 64), n_g=_log(rng, 1500, 11800), n_s=rng.randint(1, 8),
                    precision=rng.choice(["fp64", "fp32", "bf16x3"]), interstitial="fft", n_cols=rng.randint(1, 24))
    return dict(op="zgemm", m=_log(rng, 200, 10000), n=rng.randint(1, 200), k=_log(rng, 100, 6000), trans=rng.randint(0, 1))


# ------------------------------------------------------------------ inputs

def _gen(seed, role):
    return torch.Generator(device="cuda").manual_seed(1_000_003 * (int(seed) + 1) + role)


def _cn(shape, g):
    """Complex normal with E|z|^2 = 1."""
    z = torch.randn(tuple(shape) + (2,), generator=g, device="cuda", dtype=torch.float64)
    return torch.view_as_complex(z) * math.sqrt(0.5)


def _hermitian(n, m, lo, hi, g):
    """n Hermitian m x m blocks with the spectrum inside [lo, hi]."""
    z = _cn((n, m, m), g)
    w = (z + z.mH) * 0.5
    w = w / torch.linalg.matrix_norm(w, 1, keepdim=True).clamp_min(1e-300) * math.sqrt(m) * 0.4
    return 0.5 * (lo + hi) * torch.eye(m, device="cuda", dtype=w.dtype) + 0.5 * (hi - lo) * w


def _table(recip, ext, amp, g):
    """A Hermitian table v_g (v_-g = conj v_g) with a Gaussian envelope over the box |g_i| <= ext_i."""
    r = [torch.arange(-e, e + 1, device="cuda", dtype=torch.float64) for e in ext]
    gi = torch.stack(torch.meshgrid(*r, indexing="ij"), dim=-1)
    gc = gi @ torch.as_tensor(recip, device="cuda")
    z = _cn(gi.shape[:-1], g)
    return amp * torch.exp(-(gc * gc).sum(-1) / 4.0) * 0.5 * (z + torch.flip(z, (0, 1, 2)).conj())


def _gset(recip, kc, n_g):
    """The n_g integer triples of the shortest |G + k|, lexicographically ordered."""
    gmax = (3.0 * n_g * abs(np.linalg.det(recip)) / (4.0 * math.pi)) ** (1.0 / 3.0)
    lat = 2.0 * math.pi * np.linalg.inv(recip).T
    nmax = [int(math.ceil(1.3 * gmax * np.linalg.norm(lat[i]) / (2 * math.pi))) + 2 for i in range(3)]
    r = [torch.arange(-m, m + 1, device="cuda") for m in nmax]
    ints = torch.stack(torch.meshgrid(*r, indexing="ij"), dim=-1).reshape(-1, 3)
    cart = ints.double() @ torch.as_tensor(recip, device="cuda") + torch.as_tensor(kc, device="cuda")
    len2 = torch.round((cart * cart).sum(-1) * 1e9)  # ties at the cut in lexicographic order
    sel = torch.sort(torch.sort(len2, stable=True).indices[:n_g]).values
    return ints[sel].to(torch.int32), cart[sel].contiguous()


def _good(n):
    """The smallest 2^a 3^b 5^c at or above n."""
    while True:
        m = n
        for p in (2, 3, 5):
            while m % p == 0:
                m //= p
        if m == 1:
            return n
        n += 1


class Physics:
    """A drawn system on the GPU and the method's plain 64-bit arithmetic on it, k-point by k-point."""

    def __init__(self, case, seed):
        self.case = c = case
        lat = LATTICES[c["lattice"]]
        self.omega = abs(float(np.linalg.det(lat)))
        self.recip = 2.0 * math.pi * np.linalg.inv(lat).T
        nk, na, self.na = c["n_k"], c["n_atoms"], 2 * (c["lmax"] + 1) ** 2
        self.m = self.na + c["n_lo"]
        self.nlo = na * c["n_lo"]
        # unequal k-points: the sizes fall by about an eighth from one to the next
        self.ng = [max(int(c["n_g"] * (1.0 - 0.123 * k)), 1) for k in range(nk)]
        kcs = [np.array([0.25 * k, 0.25 * (k // 2), 0.0]) @ self.recip for k in range(nk)]
        sets = [_gset(self.recip, kcs[k], self.ng[k]) for k in range(nk)]
        self.gint, self.gk = [s[0] for s in sets], [s[1] for s in sets]
        self.ext = [max(int((gi[:, i].max() - gi[:, i].min()).item()) for gi in self.gint) for i in range(3)]
        self.F = [_good(2 * e + 1) for e in self.ext]
        self.vtab = _table(self.recip, self.ext, 0.1, _gen(seed, 1))
        g = _gen(seed, 2)
        self.h = _hermitian(na, self.m, -1.0, 1.0, g)
        self.o = _hermitian(na, self.m, 0.5, 2.0, g)
        self.p = _hermitian(3 * na, self.m, -0.5, 0.5, g).reshape(na, 3, self.m, self.m)
        self.amat, self.X, self.eps, self.P = [], [], [], []
        vr = self.image(self.vtab)
        self.vr = vr
        for k in range(nk):
            g = _gen(seed, 10 + k)
            g2 = (self.gk[k] ** 2).sum(-1)
            # stored as (n_g, rows): the column-major image of the rows x n_g block
            self.amat.append(_cn((self.ng[k], na * self.na), g) * (torch.exp(-g2 / 20.0) / math.sqrt(self.ng[k]))[:, None])
            x = _cn((self.ng[k] + self.nlo, c["n_aux"]), g)
            x[: self.ng[k]] *= torch.exp(-g2 / (0.5 * g2.max()))[:, None]
            x[self.ng[k]:] *= 0.3
            # the ground-state basis: S-orthonormal Ritz vectors of H0 in the span of x
            for _ in range(2):
                sx = self.mt(k, x, self.o, x)
                r = torch.linalg.cholesky(self.hermitise(x.mH @ sx)).mH
                x = torch.linalg.solve_triangular(r, x, upper=True, left=False)
            hx = self.h0(k, x)
            e, v = torch.linalg.eigh(self.hermitise(x.mH @ hx))
            x = x @ v
            t = x.sum(0)  # the context's convention: each vector's entries add up to a positive number
            x = x * (t.conj() / t.abs())
            self.X.append(x)
            self.eps.append(e)

    @staticmethod
    def hermitise(a):
        return 0.5 * (a + a.mH)

    def local(self, k, x):
        """[A_a x_G ; x_lo(a)] of every atom: (atoms, m, columns)."""
        na, n = self.case["n_atoms"], x.shape[1]
        q = (self.amat[k].T @ x[: self.ng[k]]).reshape(na, self.na, n)
        return torch.cat([q, x[self.ng[k]:].reshape(na, -1, n)], dim=1)

    def mt(self, k, x, blocks, pw, loc=None):
        """sum_a E_a^H block_a E_a x, with the plane-wave rows of `pw` added (the interstitial part)."""
        y = blocks @ (self.local(k, x) if loc is None else loc)
        n = x.shape[1]
        out = torch.cat([self.amat[k].conj() @ y[:, : self.na].reshape(-1, n), y[:, self.na:].reshape(-1, n)])
        out[: self.ng[k]] += pw[: self.ng[k]]
        return out

    def box(self, tab):
        b = torch.zeros(self.F, device="cuda", dtype=torch.complex128)
        i = [torch.arange(-e, e + 1, device="cuda") % f for e, f in zip(self.ext, self.F)]
        b[i[0][:, None, None], i[1][None, :, None], i[2][None, None, :]] = tab
        return b

    def image(self, tab):
        """v(r) = sum_d v_d e^{2 pi i d r / F}."""
        return torch.fft.ifftn(self.box(tab)) * float(np.prod(self.F))

    def scatter(self, k, x):
        i = self.gint[k].long() % torch.as_tensor(self.F, device="cuda")
        lin = (i[:, 0] * self.F[1] + i[:, 1]) * self.F[2] + i[:, 2]
        b = torch.zeros((x.shape[1], int(np.prod(self.F))), device="cuda", dtype=torch.complex128)
        b[:, lin] = x[: self.ng[k]].T
        return b.reshape([-1] + self.F), lin

    def conv(self, k, x, vr, chunk=32):
        """sum_G' v_{G-G'} x_G' on a grid without aliasing."""
        out = []
        for c0 in range(0, x.shape[1], chunk):
            b, lin = self.scatter(k, x[:, c0: c0 + chunk])
            b = torch.fft.fftn(torch.fft.ifftn(b, dim=(1, 2, 3)) * vr, dim=(1, 2, 3))
            out.append(b.reshape(b.shape[0], -1)[:, lin].T)
        return torch.cat(out, dim=1)

    def h0(self, k, x):
        g2 = 0.5 * (self.gk[k] ** 2).sum(-1)
        return self.mt(k, x, self.h, g2[:, None] * x[: self.ng[k]] + self.conv(k, x, self.vr))

    def operator(self, k, x, a, dvr=None, dh=None):
        """H(A) x, S x and c^H P_l c per column, from the submatrices."""
        loc = self.local(k, x)
        sx = self.mt(k, x, self.o, x, loc)
        blocks = self.h if dh is None else self.h + dh
        g2 = 0.5 * (self.gk[k] ** 2).sum(-1)
        vr = self.vr if dvr is None else self.vr + dvr
        hx = self.mt(k, x, blocks, g2[:, None] * x[: self.ng[k]] + self.conv(k, x, vr), loc)
        pv = []
        for l in range(3):
            px = self.mt(k, x, self.p[:, l], self.gk[k][:, l, None] * x[: self.ng[k]], loc)
            hx = hx + (float(a[l]) / C_LIGHT) * px
            pv.append((x.conj() * px).sum(0).real)
        return hx + float(np.dot(a, a)) / (2 * C_LIGHT ** 2) * sx, sx, torch.stack(pv)

    def momentum(self, k):
        x = self.X[k]
        loc = self.local(k, x)
        return torch.stack([self.hermitise(x.mH @ self.mt(k, x, self.p[:, l], self.gk[k][:, l, None] * x[: self.ng[k]], loc))
                            for l in range(3)])

    def system(self):
        """The dict that Context takes (host arrays)."""
        c, na = self.case, self.case["n_atoms"]
        host = lambda t: t.cpu().numpy()  # noqa: E731
        return dict(
            n_k=c["n_k"], n_s=c["n_s"], n_aux=c["n_aux"], n_atoms=na, omega=self.omega, c_light=C_LIGHT, recip=self.recip,
            occ=np.full(c["n_s"], 2.0), wk=np.full(c["n_k"], 1.0 / c["n_k"]), dt=c["dt"],
            n_g=np.array(self.ng, dtype=np.int32), n_a=np.full(na, self.na, dtype=np.int32),
            n_lo=np.full(na, c["n_lo"], dtype=np.int32), g_int=[host(g) for g in self.gint], gk=[host(g) for g in self.gk],
            amat=[host(t).T for t in self.amat], h=list(host(self.h)), o=list(host(self.o)), p=list(host(self.p)),
            vt_dim=np.array([2 * e + 1 for e in self.ext], dtype=np.int32), vtab=host(self.vtab))


def _drive(case, seed):
    """Pulse samples (a strong pulse near its peak), potential-change scales and the starting states."""
    n, dt = case["steps"], case["dt"]
    r = np.random.Generator(np.random.PCG64([int(seed), 77]))
    t = r.uniform(5.0, 50.0) + (np.arange(n) + 0.5) * dt
    e = r.standard_normal(3)
    a = 5.0 * np.sin(0.3 * t)[:, None] * (e / np.linalg.norm(e))[None, :]
    s = np.sin(0.1 * t) if case.get("drive") == "dv" else None
    return np.ascontiguousarray(a), s


def _theta(case, seed):
    """Orthonormal states in mid-run: mostly the occupied ones, a tenth of their charge excited."""
    out = []
    for k in range(case["n_k"]):
        z = 0.3 / math.sqrt(case["n_aux"]) * _cn((case["n_aux"], case["n_s"]), _gen(seed, 40 + k))
        z[: case["n_s"]] += torch.eye(case["n_s"], device="cuda", dtype=z.dtype)
        r = torch.linalg.cholesky(z.mH @ z).mH
        out.append(torch.linalg.solve_triangular(r, z, upper=True, left=False))
    return out


def _dv(ph, seed):
    g = _gen(seed, 60)
    return _hermitian(ph.case["n_atoms"], ph.m, -1e-2, 1e-2, g), _table(ph.recip, ph.ext, 1e-2, g)


def _zgemm_inputs(case, seed):
    g = _gen(seed, 5)
    m, n, k = case["m"], case["n"], case["k"]
    rows, cols = (k, m) if case["trans"] else (m, k)
    # column-major operands: the transposes of contiguous tensors
    return _cn((cols, rows), g), _cn((n, k), g) / math.sqrt(k)


# ------------------------------------------------------------------ the calls

def prepare(case, seed):
    if case["op"] == "zgemm":
        a, x = _zgemm_inputs(case, seed)
        return dict(case=case, a=a, x=x, c=torch.zeros((case["n"], case["m"]), device="cuda", dtype=torch.complex128))
    ph = Physics(case, seed)
    sysd = ph.system()
    sysd["caux"] = [t.T.contiguous().cpu().numpy().T for t in ph.X]
    kw = {}
    if case.get("drive") == "hartree":
        c0 = [(x @ t).T.contiguous().cpu().numpy().T for x, t in zip(ph.X, _theta(case, seed))]
        kw = dict(hartree=True, hartree_bound=50.0, hartree_mt_u=case["mt_u"], c0=c0)
    # the program's own stream: its tensors and the context's work are ordered on it
    stream = torch.cuda.Stream()
    ctx = Context(sysd, stream=stream.cuda_stream, precision=case["precision"], interstitial=case["interstitial"],
                  graph_steps=case.get("graph", 1), max_record=256, a_max=6.0, s_max=1.0, **kw)
    st = dict(case=case, ctx=ctx, stream=stream)
    if case["op"] == "apply":
        g = _gen(seed, 50)
        st["x"] = (_cn((case["n_cols"], ph.ng[0] + ph.nlo), g) / math.sqrt(ph.ng[0])).contiguous()
        st["a"] = np.array([1.0, -2.0, 3.0])
        return st
    st["a"], st["s"] = _drive(case, seed)
    if case.get("drive") == "dv":
        dh, dvt = _dv(ph, seed)
        ctx.set_dv(dict(dh=list(dh.cpu().numpy()), dvtab=dvt.cpu().numpy()))
    if case.get("drive") != "hartree":
        for k, t in enumerate(_theta(case, seed)):
            ctx.set_state(k, t.cpu().numpy())
    if case["op"] == "adjoint":
        st["g"] = np.random.Generator(np.random.PCG64([int(seed), 78])).standard_normal(3)
    return st


def _keep(case, record, theta):
    """What the program keeps: the form's accuracy decides the type (see the top of this file)."""
    out = {n: record[n] for n in ("t", "dt_cr", "j", "dmu", "n_exc", "energy", "j_full")}
    low = case["precision"] != "fp64"
    for n in ("energy", "j_full") + (("j", "dmu", "n_exc") if case["drive"] != "field" else ()):
        if low and out[n] is not None:
            out[n] = out[n].astype(np.float32)
    out["theta"] = [t.astype(np.complex64) if low and case["drive"] != "field" else t for t in theta]
    return out


def run(state):
    case = state["case"]
    if case["op"] == "zgemm":
        a, x, c = state["a"], state["x"], state["c"]
        rttddft.rttddft_zgemm_bf16x3(case["trans"], case["m"], case["n"], case["k"], a, a.shape[1], x, x.shape[1], c, c.shape[1])
        return c.to(torch.complex64)
    ctx = state["ctx"]
    if case["op"] == "apply":
        # the block is column-major: a contiguous (columns, rows) tensor
        x = state["x"]
        with torch.cuda.stream(state["stream"]):
            hx, sx = torch.empty_like(x), torch.empty_like(x)
            rttddft.rttddft_apply(ctx.ctx, 0, case["n_cols"], x, state["a"], 0.0, hx, sx)
            return (hx, sx) if case["precision"] == "fp64" else (hx.to(torch.complex64), sx.to(torch.complex64))
    if case["op"] == "adjoint":
        return ctx.adjoint(state["a"], state["g"], ckpt_every=case["ckpt"])
    ctx.step(state["a"], state["s"])
    return _keep(case, ctx.observables(), [ctx.get_state(k) for k in range(case["n_k"])])


# ------------------------------------------------------------------ 64-bit results

def _expm_apply(h, theta, dt):
    """exp(-i dt h) theta by its Taylor series in equal parts of norm below 1."""
    parts = max(1, int(math.ceil(dt * float(torch.linalg.matrix_norm(h.detach(), 1)))))
    for _ in range(parts):
        term, out = theta, theta
        for n in range(1, 24):
            term = (-1j * dt / parts / n) * (h @ term)
            out = out + term
        theta = out
    return theta


def _hsub(ph, pp, k, a):
    """The subspace Hamiltonian at vector potential a (a tensor)."""
    h = torch.diag(ph.eps[k]).to(torch.complex128) + torch.einsum("l,lij->ij", (a / C_LIGHT).to(torch.complex128), pp[k])
    return h + (a @ a) / (2 * C_LIGHT ** 2) * torch.eye(h.shape[0], device="cuda", dtype=h.dtype)


def _current(ph, pp, theta, a, wk):
    j = 0
    for k, th in enumerate(theta):
        pt = torch.einsum("lij,js->lis", pp[k], th)
        val = (th.conj()[None] * pt).sum((1, 2)).real + a / C_LIGHT * (th.conj() * th).sum().real
        j = j - wk * 2.0 / ph.omega * val
    return j


def _density(ph, c, wk):
    """The interstitial density's coefficients n_g on the table box."""
    n = torch.zeros(ph.F, device="cuda", dtype=torch.float64)
    vol = float(np.prod(ph.F))
    for k, ck in enumerate(c):
        b, _ = ph.scatter(k, ck)
        n += 2.0 * wk * (torch.fft.ifftn(b, dim=(1, 2, 3)) * vol).abs().square().sum(0)
    f = torch.fft.fftn(n) / vol / ph.omega
    i = [torch.arange(-e, e + 1, device="cuda") % q for e, q in zip(ph.ext, ph.F)]
    return f[i[0][:, None, None], i[1][None, :, None], i[2][None, None, :]]


def _mt_density(ph, c, wk):
    return sum(2.0 * wk * (loc := ph.local(k, ck)) @ loc.mH for k, ck in enumerate(c))


def exact(case, seed):
    if case["op"] == "zgemm":
        a, x = _zgemm_inputs(case, seed)
        return x @ (a.conj().T if case["trans"] else a)
    ph = Physics(case, seed)
    nk, wk, dt = case["n_k"], 1.0 / case["n_k"], case["dt"]
    if case["op"] == "apply":
        x = (_cn((case["n_cols"], ph.ng[0] + ph.nlo), _gen(seed, 50)) / math.sqrt(ph.ng[0])).T
        hx, sx, _ = ph.operator(0, x, np.array([1.0, -2.0, 3.0]))
        return hx.T.contiguous(), sx.T.contiguous()
    a_all, s_all = _drive(case, seed)
    pp = [ph.momentum(k) for k in range(nk)]
    eye = torch.eye(case["n_aux"], case["n_s"], device="cuda", dtype=torch.complex128)
    theta = _theta(case, seed)
    start = theta if case.get("drive") == "hartree" else [eye] * nk  # the state at set-up
    j_gs = _current(ph, pp, start, torch.zeros(3, device="cuda", dtype=torch.float64), wk)
    if case["op"] == "adjoint":
        g = torch.as_tensor(np.random.Generator(np.random.PCG64([int(seed), 78])).standard_normal(3), device="cuda")
        a = torch.as_tensor(a_all, device="cuda").requires_grad_(True)
        dmu, jp = 0, torch.zeros(3, device="cuda", dtype=torch.float64)
        for i in range(len(a_all)):
            theta = [_expm_apply(_hsub(ph, pp, k, a[i]), theta[k], dt) for k in range(nk)]
            j = _current(ph, pp, theta, a[i], wk) - j_gs
            dmu, jp = dmu + ph.omega * dt * 0.5 * (jp + j), j
        (g @ dmu).backward()
        return a.grad.cpu().numpy(), dmu.detach().cpu().numpy()
    dh1 = dv1 = None
    if case["drive"] == "dv":
        dh1, dvt = _dv(ph, seed)
        dv1 = ph.image(dvt)
    if case["drive"] == "hartree":
        c0 = [ph.X[k] @ theta[k] for k in range(nk)]
        n0, m0 = _density(ph, c0, wk), _mt_density(ph, c0, wk)
        r = [torch.arange(-e, e + 1, device="cuda", dtype=torch.float64) for e in ph.ext]
        g2 = ((torch.stack(torch.meshgrid(*r, indexing="ij"), dim=-1) @ torch.as_tensor(ph.recip, device="cuda")) ** 2).sum(-1)
        kern = torch.where(g2 > 0, 4 * math.pi / torch.where(g2 > 0, g2, 1.0), 0.0)
        c = c0
    rec = {n: [] for n in ("j", "dmu", "n_exc", "energy", "j_full")}
    dmu, jp = np.zeros(3), np.zeros(3)
    zero = lambda k: torch.zeros((ph.ng[k], case["n_aux"]), device="cuda", dtype=torch.complex128)  # noqa: E731
    dvv = None if dv1 is None else [ph.hermitise(ph.X[k].mH @ ph.mt(k, ph.X[k], dh1, ph.conv(k, ph.X[k], dv1))) for k in range(nk)]
    for i, a in enumerate(a_all):
        dvr = dh = None
        if case["drive"] == "dv":
            dvr, dh = float(s_all[i]) * dv1, float(s_all[i]) * dh1
        elif case["drive"] == "hartree":
            dvr = ph.image(kern * (_density(ph, c, wk) - n0))
            dh = case["mt_u"] * (_mt_density(ph, c, wk) - m0)
        at = torch.as_tensor(a, device="cuda")
        for k in range(nk):
            h = _hsub(ph, pp, k, at)
            if dvv is not None:
                h = h + float(s_all[i]) * dvv[k]
            elif dvr is not None:
                x = ph.X[k]
                h = h + ph.hermitise(x.mH @ ph.mt(k, x, dh, ph.conv(k, x, dvr)))
            theta[k] = _expm_apply(h, theta[k], dt)
        c = [ph.X[k] @ theta[k] for k in range(nk)]
        e, jf, nx = 0.0, torch.zeros(3, device="cuda", dtype=torch.float64), 2.0 * case["n_s"]
        for k in range(nk):
            hx, sx, pv = ph.operator(k, c[k], a, dvr, dh)
            e += 2.0 * wk * float((c[k].conj() * hx).sum().real)
            norm = (c[k].conj() * sx).sum().real
            jf = jf - 2.0 * wk / ph.omega * (pv.sum(1) + at / C_LIGHT * norm)
            nx -= 2.0 * wk * float(theta[k][: case["n_s"]].abs().square().sum())
        j = _current(ph, pp, theta, at, wk)
        jind = (j - j_gs).cpu().numpy()
        dmu = dmu + ph.omega * dt * 0.5 * (jp + jind)
        jp = jind
        for n, v in (("j", j.cpu().numpy()), ("dmu", dmu), ("n_exc", nx), ("energy", e), ("j_full", jf.cpu().numpy())):
            rec[n].append(v)
    out = {n: np.array(v) for n, v in rec.items()}
    # the times are a product and dt_cr comes from the bounds of the spectrum that the propagator took
    out.update(t=None, dt_cr=None, theta=[t.cpu().numpy() for t in theta])
    return out


# ------------------------------------------------------------------ work

def work(case):
    """Inputs read once and outputs written once, and the flops of the method in its submatrix form."""
    if case["op"] == "zgemm":
        m, n, k = case["m"], case["n"], case["k"]
        return dict(bytes=16 * (m * k + n * k + m * n) + 8 * m * n, flops=8 * m * n * k)
    w = 16 if case["precision"] == "fp64" else 8  # bytes of a stored complex number of the form
    ns, nx = case["n_s"], case["n_aux"]
    na = 2 * (case["lmax"] + 1) ** 2
    ma, m, nat = case["n_atoms"] * na, na + case["n_lo"], case["n_atoms"]
    cols = case["n_cols"] if case["op"] == "apply" else ns
    size, flops, out = 0, 0, 0
    for k in range(case["n_k"]):
        ng = max(int(case["n_g"] * (1.0 - 0.123 * k)), 1)
        nb = ng + nat * case["n_lo"]
        fft = 10 * 8 * ng * math.log2(8 * ng)  # the interstitial sum of one column by transforms on about 8 N_G points
        op = cols * (8 * (3 * ma * ng + 5 * m * m * nat) + fft)
        sub = 8 * nx * nx * ns * 13 + 8 * 3 * nx * nx
        if case["op"] == "apply":
            size += w * (ma * ng + 5 * m * m * nat)
            out += 16 * 3 * nb * cols
            flops += op
            continue
        size += 16 * 3 * nx * nx
        out += 16 * 2 * nx * ns
        if case["op"] == "adjoint":
            flops += 3 * sub
            continue
        size += w * (ma * ng + nb * nx + 5 * m * m * nat)
        flops += sub + op + 8 * 2 * nb * nx * ns
        if case["drive"] != "field":
            # CC^H dV CC: the blocks on the local coordinates, the interstitial sum of every auxiliary vector
            flops += 8 * nat * m * nx * (m + nx) + nx * fft + 8 * nx * nx * ng
    steps = case.get("steps", 1)
    return dict(bytes=size + out + (8 * 16 * steps if case["op"] != "apply" else 0), flops=flops * steps)
