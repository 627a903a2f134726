"""The work a user has this library do, as timed cases: one propagation step in every precision
and size range, one Hamiltonian application, the energies and torques of a running propagation,
a differentiated step, and the stand-alone Poisson solve.

A case is a dict of plain values; ``system`` builds its atoms, cell and field table, ``prepare``
the handle and the spinors (on the GPU, from the seed), ``run`` makes one pass through the public
entry points, and ``exact`` evaluates the same result in FP64 with plain torch.
"""
import math

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

from paper_2506_21908_gb300 import _lib, autograd

PROJ = {"cuda": None, "tf32x3": _lib.PROJ_TF32X3, "bf16x3": _lib.PROJ_BF16X3, "f16x3": _lib.PROJ_F16X3}
EXP = {"chebyshev": _lib.EXP_CHEBYSHEV, "taylor": _lib.EXP_TAYLOR, "crank_nicolson": _lib.EXP_CRANK_NICOLSON}
SPIN = {"noncollinear": _lib.SPIN_NONCOLLINEAR, "collinear": _lib.SPIN_COLLINEAR}
GRIDS = (8, 12, 16, 24, 32, 48, 64, 96)
R_CUT = 5.0


def _case(name, do, geometry, n, nstates, precision="mixed", proj="cuda", **more):
    c = dict(name=name, do=do, geometry=geometry, n=n, nstates=nstates, nk=1, natoms=0, lmax=2, precision=precision,
             proj=proj, exp="chebyshev", spin="noncollinear", n_sc=1)
    c.update(more)
    return c


def listed():
    return [
        # The Poisson solve alone, for a caller with its own density loop: the smallest call there is.
        _case("hartree_48", "hartree", "bcc", 48, 0, "fp64"),
        # The tiny reference system: 24^3, four spinors, FP64 (the default precision); launches count.
        _case("tiny_step_fp64", "step", "tiny", 24, 4, "fp64", lmax=1),
        # A small molecule at two k-points with an odd number of states, FP32-mixed: latency again.
        _case("small_step_mixed", "step", "free", 32, 7, nk=2, natoms=3),
        # One H application to all spinors of the magnetic cluster in FP64, the operator's diagnostic.
        _case("cluster_apply_fp64", "apply", "cluster", 64, 104, "fp64"),
        # The magnetic cluster's step, FP32-mixed with the default (CUDA-core) projectors ...
        _case("cluster_step_mixed", "step", "cluster", 64, 104),
        # ... and with the split FP16 tensor-core projectors, the benchmark's mode.
        _case("cluster_step_f16x3", "step", "cluster", 64, 104, proj="f16x3"),
        # The bcc supercell: eight k-points with 128 spinors each on 48^3.
        _case("bcc_step_f16x3", "step", "bcc", 48, 128, proj="f16x3", nk=8),
        # The large supercell's grid and 128 atoms with an eighth of its 1024 spinors.
        _case("large_step_f16x3", "step", "large", 96, 128, proj="f16x3"),
        # An alternative propagator and spin mode, an odd number of states: Crank-Nicolson, collinear.
        _case("cn_collinear_tf32x3", "step", "cluster", 48, 27, proj="tf32x3", exp="crank_nicolson", spin="collinear"),
        # The FP64 step at production grid size, which the FP32-mixed mode is checked against.
        _case("cluster_step_fp64", "step", "cluster", 64, 13, "fp64"),
        # Loss and gradient of one step with respect to the field table (the discrete adjoint).
        _case("gradient_fp64", "gradient", "bcc", 48, 5, "fp64"),
        # What a running propagation reports: densities, energies, norms, moments and torques.
        _case("report_fp64", "report", "cluster", 64, 26, "fp64"),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    do = rng.choices(("hartree", "step", "apply", "gradient", "report"), (1, 8, 1, 1, 1))[0]
    if do == "hartree":
        c = _case("", do, "bcc", rng.choice(GRIDS[:-1]), 0, "fp64")
        c["lx"], c["ly"] = round(rng.uniform(8.0, 24.0), 3), round(rng.uniform(8.0, 24.0), 3)
    else:
        mixed = do == "step" and rng.random() < 0.8
        n = rng.choice(GRIDS[1:] if mixed or do == "apply" else GRIDS[:-1])
        geometry = rng.choice(("free", "cluster", "bcc") if n >= 24 else ("free",))
        nk = {"bcc": 8, "cluster": 1, "free": rng.choice((1, 2, 3))}[geometry]
        # components x points no costlier than the largest listed case, by kind and precision
        most = {"step": 1.2e8 if mixed else 6.0e6, "apply": 2.5e7, "gradient": 2.0e6, "report": 1.2e7}[do]
        top = max(1, min(150, int(most / (2 * nk * n ** 3))))
        proj = rng.choice(("cuda", "f16x3", "f16x3", "bf16x3", "tf32x3") if mixed and n % 16 == 0 else ("cuda",))
        c = _case("", do, geometry, n, _log_int(rng, 1, top), "mixed" if mixed else "fp64", proj, nk=nk,
                  natoms=rng.randint(1, 5), lmax=rng.choice((1, 2, 2)), n_sc=rng.choice((1, 1, 2)))
        if do == "step":
            c["exp"] = rng.choices(tuple(EXP), (6, 1, 1))[0]
            c["spin"] = rng.choices(tuple(SPIN), (5, 1))[0]
    del c["name"]
    return c


# ----------------------------------------------------------------------------- inputs

def system(case, seed):
    """Atoms, cell, k-points, occupations and field table (numpy, atomic units)."""
    rng = np.random.default_rng(seed)
    g, n = case["geometry"], case["n"]
    Z, dt, r_cut = 8.0, 0.04, R_CUT
    kpts = np.zeros((1, 3))
    if g == "tiny":
        L, dt = np.full(3, 10.0), 0.05
        pos = np.full((1, 3), 5.0)
    elif g == "cluster":
        L = np.full(3, 24.0)
        phi = 0.5 * (1.0 + math.sqrt(5.0))
        v = np.array([w for a in (-1.0, 1.0) for b in (-phi, phi) for w in ((0, a, b), (a, b, 0), (b, 0, a))])
        pos = np.vstack([np.zeros(3), 4.7 * v / np.linalg.norm(v[0])]) + 12.0
    elif g in ("bcc", "large"):
        reps, a = (2, 5.42) if g == "bcc" else (4, 5.425)
        L = np.full(3, reps * a)
        cells = np.array([[i, j, k] for i in range(reps) for j in range(reps) for k in range(reps)], np.float64)
        pos = np.concatenate([cells, cells + 0.5]) * a
        if case["nk"] == 8:
            q = 0.5 * math.pi / L[0]
            kpts = np.array([[x * q, y * q, z * q] for x in (-1, 1) for y in (-1, 1) for z in (-1, 1)])
    else:
        L, Z, dt, r_cut = np.full(3, 9.0), 3.0, 0.05, 4.0
        pos = rng.uniform(0.0, 9.0, (case["natoms"], 3))
        if case["nk"] > 1:
            kpts = rng.uniform(-0.3, 0.3, (case["nk"], 3))
    if "lx" in case:
        L = np.array([case["lx"], case["ly"], L[2]])
    if g != "tiny":
        pos = np.mod(pos + rng.normal(0.0, 0.1, pos.shape), L)
    lmax = case["lmax"]
    D = np.array([[1.0, 0.5, 0.25]])[:, :lmax + 1]
    lam = np.full((1, lmax + 1), 0.02 if case["spin"] == "noncollinear" and g != "tiny" else 0.0)
    lam[:, 0] = 0.0
    nk, nst = len(kpts), max(1, case["nstates"])
    occ = np.ones((nk, nst))
    if g == "free":
        occ[:, -1] = 0.5
    # the laser A = -int E dt of a pulse under way, in velocity gauge, and a static B
    t = dt * np.arange(5)
    A = np.zeros((5, 3)) if g == "tiny" else -(0.01 / 0.057) * np.sin(0.057 * (t + rng.uniform(5.0, 20.0)))[:, None] * np.array([1.0, 0.0, 0.0])
    B = np.tile([0.0, 0.0, 0.0] if g in ("tiny", "cluster", "large") else [0.02, -0.01, 0.03] if g == "free" else [0.001, 0.0, 0.0], (5, 1))
    return dict(L=L, n=n, pos=pos, species=np.zeros(len(pos), np.int32), Z=np.array([Z]), rc=np.array([0.8]),
                width=np.array([1.0]), lmax=lmax, D=D, lam=lam, r_cut=min(r_cut, 0.5 * L.min()), kpts=kpts,
                kw=np.full(nk, 1.0 / nk), occ=occ, dt=dt, t=t, A=A, B=B)


def _grid(s):
    """Coordinates of the grid points per axis, on the GPU."""
    return [torch.arange(s["n"], device="cuda", dtype=torch.float64) * (s["L"][a] / s["n"]) for a in range(3)]


def spinors(case, s, seed, dtype):
    """Orthonormal spinors [k][state][2][z][y][x]: s, p and d Gaussians with random complex weights
    and the atom's spin axis, or smooth random fields where there are more states than orbitals."""
    n, L, nk, nst = s["n"], s["L"], len(s["kpts"]), s["occ"].shape[1]
    gen = torch.Generator(device="cuda").manual_seed(1000 + seed)
    dV = float(np.prod(L)) / n ** 3
    out = torch.empty((nk, nst, 2, n, n, n), dtype=dtype, device="cuda")
    real = torch.float64 if dtype == torch.complex128 else torch.float32
    atoms = case["geometry"] not in ("tiny", "free") and nst <= 8 * len(s["pos"])
    xs = _grid(s)
    for k in range(nk):
        for i in range(nst):
            if atoms:
                a = i % len(s["pos"])
                d = [x - s["pos"][a, ax] for ax, x in enumerate(xs)]
                d = [v - L[ax] * torch.round(v / L[ax]) for ax, v in enumerate(d)]
                g = [torch.exp(-0.5 * v * v) for v in d]
                w = torch.randn((3, 3, 3), dtype=torch.complex128, device="cuda", generator=gen)
                p = torch.arange(3, device="cuda")
                w = w * (p[:, None, None] + p[None, :, None] + p[None, None, :] <= 2)
                f = [torch.stack([v ** q * u for q in range(3)]).to(torch.complex128) for v, u in zip(d, g)]
                phi = torch.einsum("abc,az,by,cx->zyx", w, f[2], f[1], f[0])
                q = [torch.exp(-1j * float(s["kpts"][k, ax]) * x) for ax, x in enumerate(xs)]
                phi = phi * q[2][:, None, None] * q[1][None, :, None] * q[0][None, None, :]
                th = (0.35 if a == 1 else 0.05) + (math.pi if i % 8 >= 5 else 0.0)
                chi = (math.cos(0.5 * th), math.sin(0.5 * th))
                for c in range(2):
                    out[k, i, c] = (chi[c] * phi).to(dtype)
            else:
                f = torch.randn((2, n, n, n), dtype=torch.complex128, device="cuda", generator=gen)
                q = torch.fft.fftfreq(n, device="cuda", dtype=torch.float64) ** 2
                f = torch.fft.ifftn(torch.fft.fftn(f, dim=(1, 2, 3)) * torch.exp(-(q[:, None, None] + q[:, None] + q) / 0.08), dim=(1, 2, 3))
                out[k, i] = f.to(dtype)
        v = out[k].reshape(nst, -1)
        S = (v.conj() @ v.T).to(torch.complex128) * dV
        w, U = torch.linalg.eigh(S)
        M = (U * w.clamp_min(1e-6 * float(w[-1])).rsqrt()) @ U.mH
        out[k] = (M.T.to(dtype) @ v).reshape(out[k].shape)
    return out if real is torch.float64 else out.contiguous()


def _density_input(case, s, seed):
    """A smooth positive density for the stand-alone Poisson solve."""
    gen = torch.Generator(device="cuda").manual_seed(2000 + seed)
    rho = torch.zeros((case["n"],) * 3, dtype=torch.float64, device="cuda")
    for R in s["pos"]:
        g = []
        for ax, x in enumerate(_grid(s)):
            d = x - R[ax]
            g.append(torch.exp(-0.5 * (d - s["L"][ax] * torch.round(d / s["L"][ax])) ** 2))
        rho += torch.rand((), dtype=torch.float64, device="cuda", generator=gen) * g[2][:, None, None] * g[1][:, None] * g[0]
    return rho


def prepare(case, seed):
    s = system(case, seed)
    if case["do"] == "hartree":
        rho = _density_input(case, s, seed)
        return dict(do="hartree", rho=rho, out=torch.empty_like(rho), L=s["L"])
    fp64 = case["precision"] == "fp64"
    h = _lib.TDDFT(s["L"], s["n"], s["pos"], s["species"], s["Z"], s["rc"], s["width"], s["lmax"], s["D"], s["lam"],
                   s["r_cut"], s["kpts"], s["kw"], s["occ"], s["dt"],
                   precision=_lib.FP64 if fp64 else _lib.FP32_MIXED, proj_mode=PROJ[case["proj"]],
                   exp_kind=EXP[case["exp"]], n_sc=case["n_sc"], spin_mode=SPIN[case["spin"]])
    h.set_fields(s["t"], s["A"], s["B"])
    psi = spinors(case, s, seed, torch.complex128 if fp64 else torch.complex64)
    st = dict(do=case["do"], h=h, psi=psi, out=torch.empty_like(psi))
    if case["do"] in ("apply", "report"):
        h.set_states(psi, 0.0)
    if case["do"] == "gradient":
        st["seed"] = autograd.mz_seed(s["n"], s["L"])
    return st


def run(state):
    do = state["do"]
    if do == "hartree":
        _lib.hartree_noalloc(state["rho"], state["out"], state["L"])
        return state["out"]
    h = state["h"]
    if do == "step":
        h.set_states(state["psi"], 0.0)
        h.step(1)
        return h.get_states(state["out"])
    if do == "apply":
        return h.apply_hamiltonian(state["psi"], state["out"])
    if do == "gradient":
        h.set_states(state["psi"], 0.0)
        loss, dA, dB = h.backward(1, state["seed"], ckpt_every=1)
        return dict(loss=loss, dA=dA, dB=dB, psi=h.get_states(state["out"]))
    n, m, E, norms = h.observables()
    M, N = h.atom_moments()
    T = h.torques()
    # the XC torque is zero in the locally collinear approximation (its rounding enters the total)
    return dict(n=n, m=m, norms=norms, moments=M, electrons=N, soc=T["soc"], torque=T["total"],
                E=[E[k] for k in ("kin", "nl", "loc", "H", "xc", "total", "xc_pot", "N")], M=E["M"])


# ----------------------------------------------------------------------------- work

def _applies(case):
    """H applications of one pass (the Chebyshev orders of this library's systems, rounded)."""
    n, fp64 = case["n"], case["precision"] == "fp64"
    if case["do"] in ("apply", "report"):
        return 1
    if case["exp"] == "taylor":
        return 8 + 4 * (1 + case["n_sc"])
    full, half = (27, 20) if fp64 else (20, 14)
    scale = 3 if case["exp"] == "crank_nicolson" else 1
    steps = scale * (full + half * (1 + case["n_sc"])) * (n / 96.0 if case["geometry"] == "free" else 1.0)
    return (3 if case["do"] == "gradient" else 1) * max(8.0, steps)


def work(case):
    n3 = case["n"] ** 3
    fft = 5.0 * n3 * math.log2(n3)
    if case["do"] == "hartree":
        return dict(bytes=16.0 * n3, flops=2 * fft)
    nk = case["nk"]
    spin = float(nk * case["nstates"])
    size = 16.0 if case["precision"] == "fp64" else 8.0
    s = system(case, 0)
    sphere = min(4.0 / 3.0 * math.pi * s["r_cut"] ** 3 / float(np.prod(s["L"])), 1.0) * n3 * len(s["pos"])
    h = 2 * spin * (2 * fft + 40.0 * n3 + 8.0 * (case["lmax"] + 1) ** 2 * sphere)
    psi = 2 * spin * n3 * size
    return dict(bytes=psi * (1 if case["do"] == "report" else 2) + (48.0 * n3 if case["do"] == "report" else 0.0),
                flops=_applies(case) * h)


# ----------------------------------------------------------------------------- the same in 64 bits

class _Exact:
    """The Hamiltonian, its potential and the ETRS step in FP64 with plain torch."""

    PW92 = ((0.031091, 0.21370, 7.5957, 3.5876, 1.6382, 0.49294), (0.015545, 0.20548, 14.1189, 6.1977, 3.3662, 0.62517),
            (0.016887, 0.11125, 10.357, 3.6231, 0.88026, 0.49671))

    def __init__(self, case, s):
        self.case, self.s, n = case, s, s["n"]
        self.n, self.dV = n, float(np.prod(s["L"])) / n ** 3
        f = torch.fft.fftfreq(n, device="cuda", dtype=torch.float64) * n
        self.g = [2.0 * math.pi / s["L"][a] * f for a in range(3)]
        self.G2 = self.g[2][:, None, None] ** 2 + self.g[1][:, None] ** 2 + self.g[0] ** 2
        self.coulomb = torch.where(self.G2 > 0, 4.0 * math.pi / self.G2.clamp_min(1e-300), torch.zeros_like(self.G2))
        if case["do"] == "hartree":
            return
        VG = torch.zeros((n, n, n), dtype=torch.complex128, device="cuda")
        Z, rc = float(s["Z"][0]), float(s["rc"][0])
        form = torch.where(self.G2 > 0, -Z * self.coulomb * torch.exp(-0.25 * rc * rc * self.G2), math.pi * Z * rc * rc)
        for R in s["pos"]:
            e = [torch.exp(-1j * float(R[a]) * self.g[a]) for a in range(3)]
            VG += form * (e[2][:, None, None] * e[1][:, None] * e[0])
        self.vloc = (torch.fft.ifftn(VG) * (n ** 3 / float(np.prod(s["L"])))).real
        self.wf = torch.tensor(s["kw"][:, None] * s["occ"], device="cuda")
        self._projectors()

    def _projectors(self):
        s, n, lmax, w = self.s, self.n, self.s["lmax"], float(self.s["width"][0])
        xs = _grid(s)
        self.atoms = []
        for R in s["pos"]:
            d = [x - R[a] for a, x in enumerate(xs)]
            d = [v - s["L"][a] * torch.round(v / s["L"][a]) for a, v in enumerate(d)]
            r2 = d[0] ** 2 + d[1][:, None] ** 2 + d[2][:, None, None] ** 2
            idx = torch.nonzero(r2.reshape(-1) < s["r_cut"] ** 2 * (1.0 - 1e-10))[:, 0]
            x, y, z = d[0][idx % n], d[1][(idx // n) % n], d[2][idx // (n * n)]
            rr = x * x + y * y + z * z
            c = [0.5 / math.sqrt(math.pi), math.sqrt(0.75 / math.pi), 0.5 * math.sqrt(15.0 / math.pi), 0.25 * math.sqrt(5.0 / math.pi)]
            Y = [[c[0] * torch.ones_like(x)], [c[1] * y, c[1] * z, c[1] * x],
                 [c[2] * x * y, c[2] * y * z, c[3] * (3.0 * z * z - rr), c[2] * x * z, 0.5 * c[2] * (x * x - y * y)]]
            rad = torch.exp(-0.5 * rr / (w * w))
            beta = [math.sqrt(2.0 / (math.gamma(l + 1.5) * w ** (2 * l + 3))) * rad * v for l in range(lmax + 1) for v in Y[l]]
            self.atoms.append((idx, torch.stack([x, y, z], 1), torch.stack(beta)))
        # L.S in the real harmonics: (r x grad) of the l = 1 and l = 2 polynomials, closed form through
        # the complex harmonics
        nlm = (lmax + 1) ** 2
        D = np.zeros((2 * nlm, 2 * nlm), np.complex128)
        sig = np.array([[[0, 1], [1, 0]], [[0, -1j], [1j, 0]], [[1, 0], [0, -1]]])
        for l in range(lmax + 1):
            m = np.arange(-l, l + 1)
            Lp = np.diag(np.sqrt(l * (l + 1) - m[:-1] * (m[:-1] + 1.0)), -1).astype(np.complex128)
            Lc = [0.5 * (Lp + Lp.T), -0.5j * (Lp - Lp.T), np.diag(m).astype(np.complex128)]
            U = np.zeros((2 * l + 1, 2 * l + 1), np.complex128)
            for mu in m:
                if mu > 0:
                    U[mu + l, mu + l], U[mu + l, l - mu] = (-1.0) ** int(mu) / math.sqrt(2), 1 / math.sqrt(2)
                elif mu == 0:
                    U[l, l] = 1.0
                else:
                    U[mu + l, l - mu], U[mu + l, l + mu] = (-1.0) ** int(mu) / (1j * math.sqrt(2)), -1.0 / (1j * math.sqrt(2))
            LS = sum(np.kron(U.conj() @ Lc[a] @ U.T, 0.5 * sig[a]) for a in range(3))
            o = 2 * l * l
            D[o:o + 2 * (2 * l + 1), o:o + 2 * (2 * l + 1)] = s["D"][0, l] * np.eye(2 * (2 * l + 1)) + s["lam"][0, l] * LS
        self.D = torch.tensor(D, device="cuda")
        self.torque_mats = [torch.tensor(2j * (D @ S - S @ D), device="cuda")
                            for S in (np.kron(np.eye(nlm), 0.5 * sig[a]) for a in range(3))]

    # -- density and potential
    def rho(self, psi):
        out = 0.0
        for k in range(psi.shape[0]):
            for i in range(0, psi.shape[1], 16):
                u, d, w = psi[k, i:i + 16, 0], psi[k, i:i + 16, 1], self.wf[k, i:i + 16, None, None, None]
                ud = u * d.conj()
                out = out + torch.stack([(w * (u.real ** 2 + u.imag ** 2)).sum(0), (w * (d.real ** 2 + d.imag ** 2)).sum(0),
                                         (w * ud.real).sum(0), (w * ud.imag).sum(0)])
        return out

    def hartree(self, rho):
        return torch.fft.ifftn(torch.fft.fftn(rho.to(torch.complex128)) * self.coulomb).real

    def _pw92(self, rs, row):
        A, a1, b1, b2, b3, b4 = row
        q = rs.sqrt()
        q0, q1 = -2.0 * A * (1.0 + a1 * rs), 2.0 * A * q * (b1 + q * (b2 + q * (b3 + q * b4)))
        qp = A * (b1 / q + 2.0 * b2 + 3.0 * b3 * q + 4.0 * b4 * rs)
        lg = torch.log1p(1.0 / q1)
        return q0 * lg, -2.0 * A * a1 * lg - q0 * qp / (q1 * q1 + q1)

    def lsda(self, nu, nd):
        """Slater exchange and PW92 correlation: energy density, v_up, v_down (n > 0)."""
        n = nu + nd
        third = lambda v: torch.where(v > 0, v.clamp_min(1e-300), torch.ones_like(v)).pow(1.0 / 3.0) * (v > 0)  # noqa: E731
        c6 = (6.0 / math.pi) ** (1.0 / 3.0)
        cu, cd = third(nu), third(nd)
        rs = (3.0 / (4.0 * math.pi * n)) ** (1.0 / 3.0)
        z = ((nu - nd) / n).clamp(-1.0, 1.0)
        (e0, d0), (e1, d1), (ma, dma) = (self._pw92(rs, r) for r in self.PW92)
        pz, mz = third(1.0 + z), third(1.0 - z)
        den = 2.0 ** (4.0 / 3.0) - 2.0
        f, fp, z3, z4 = ((1.0 + z) * pz + (1.0 - z) * mz - 2.0) / den, (4.0 / 3.0) * (pz - mz) / den, z ** 3, z ** 4
        c = 1.709921
        ec = e0 - ma * f * (1.0 - z4) / c + (e1 - e0) * f * z4
        drs = d0 - dma * f * (1.0 - z4) / c + (d1 - d0) * f * z4
        dz = -ma / c * (fp * (1.0 - z4) - 4.0 * z3 * f) + (e1 - e0) * (fp * z4 + 4.0 * z3 * f)
        com = ec - rs / 3.0 * drs
        ex = -0.75 * c6 * (nu * cu + nd * cd)
        return ex + n * ec, -c6 * cu + com - (z - 1.0) * dz, -c6 * cd + com - (z + 1.0) * dz

    def potential(self, rho, B):
        """The 4-vector potential [v + b_z, v - b_z, 2 b_x, -2 b_y] and its parts."""
        n, m = rho[0] + rho[1], torch.stack([2.0 * rho[2], -2.0 * rho[3], rho[0] - rho[1]])
        ok = n >= 1e-14
        if self.case["spin"] == "collinear":
            nu, nd, b_dir = rho[0], rho[1], None
        else:
            m2 = (m * m).sum(0)
            mag = torch.where(m2 > 0, m2, torch.ones_like(m2)).sqrt() * (m2 > 0)
            sm = torch.minimum(mag, n)
            nu, nd = 0.5 * (n + sm), 0.5 * (n - sm)
            b_dir = torch.where(mag > 1e-14, m / mag.clamp_min(1e-14), torch.zeros_like(m))
        one = torch.ones_like(n)
        e, vu, vd = (torch.where(ok, v, 0.0 * one) for v in self.lsda(torch.where(ok, nu, one), torch.where(ok, nd, one)))
        vbar, bm = 0.5 * (vu + vd), 0.5 * (vu - vd)
        b = torch.stack([0.0 * bm, 0.0 * bm, bm]) if b_dir is None else bm * b_dir
        vH = self.hartree(n)
        Bx = B * torch.tensor([0.0, 0.0, 1.0], device="cuda", dtype=torch.float64) if b_dir is None else B
        v, bt = self.vloc + vH + vbar, b + 0.5 * Bx[:, None, None, None]
        return torch.stack([v + bt[2], v - bt[2], 2.0 * bt[0], -2.0 * bt[1]]), dict(n=n, m=m, vH=vH, e=e, vbar=vbar, b=b)

    # -- the Hamiltonian on the spinors [states][2][z][y][x] of one k-point
    def phases(self, q):
        return [torch.exp(1j * (d @ q)) for _, d, _ in self.atoms]

    def coefficients(self, psi, phases):
        """c = <beta|psi> per atom, index (p, sigma)."""
        flat, out = psi.reshape(psi.shape[0] * 2, -1), []
        for (idx, _, beta), ph in zip(self.atoms, phases):
            v = flat[:, idx] * ph
            c = torch.stack([(v * b).sum(1) for b in beta], 1) * self.dV  # plain sums: skinny FP64 products are slow
            out.append(c.reshape(psi.shape[0], 2, -1).transpose(1, 2).reshape(psi.shape[0], -1))
        return out

    def nonlocal_part(self, psi, phases):
        res = torch.zeros((psi.shape[0] * 2, self.n ** 3), dtype=torch.complex128, device="cuda")
        for (idx, d, beta), ph, c in zip(self.atoms, phases, self.coefficients(psi, phases)):
            dc = (c @ self.D.T).reshape(psi.shape[0], -1, 2).transpose(1, 2).reshape(psi.shape[0] * 2, -1)
            v = dc[:, :1] * beta[0]
            for j in range(1, len(beta)):
                v = torch.addcmul(v, dc[:, j:j + 1], beta[j].to(torch.complex128))
            res.index_add_(1, idx, v * ph.conj())
        return res.reshape(psi.shape)

    def kinetic(self, psi, q):
        k = 0.5 * ((self.g[2] + q[2])[:, None, None] ** 2 + (self.g[1] + q[1])[:, None] ** 2 + (self.g[0] + q[0]) ** 2)
        return torch.fft.ifftn(torch.fft.fftn(psi, dim=(2, 3, 4)) * k, dim=(2, 3, 4))

    def H(self, psi, V, q, phases):
        u, d = psi[:, 0], psi[:, 1]
        bm, bp = 0.5 * (V[2] + 1j * V[3]), 0.5 * (V[2] - 1j * V[3])
        loc = torch.stack([V[0] * u + bm * d, bp * u + V[1] * d], 1)
        nl = checkpoint(self.nonlocal_part, psi, phases, use_reentrant=False) if q.requires_grad else self.nonlocal_part(psi, phases)
        return self.kinetic(psi, q) + loc + nl

    # -- exponentials: Chebyshev series of f on [lo, hi] for several functions at once
    def _series(self, psi, V, q, taus):
        case, ph = self.case, self.phases(q)
        if case["exp"] == "taylor":
            outs = []
            for tau in taus:
                term, acc = psi, psi
                for k in range(1, 5):
                    term = (-1j * tau / k) * self.H(term, V, q, ph)
                    acc = acc + term
                outs.append(acc)
            return outs
        lo, hi = self.window
        c, dl, Q = 0.5 * (lo + hi), 0.5 * (hi - lo), 4096
        cos = np.cos(0.5 * math.pi / Q * np.arange(4 * Q))  # cos(k th_j) by its exact angle modulo 2 pi
        odd = 2 * np.arange(Q) + 1
        E = c + dl * cos[odd]
        cf = []
        for tau in taus:
            f = (1 - 0.5j * tau * E) / (1 + 0.5j * tau * E) if case["exp"] == "crank_nicolson" else np.exp(-1j * tau * E)
            a = np.array([2.0 / Q * (f * cos[k * odd % (4 * Q)]).sum() for k in range(400)])
            a[0] *= 0.5
            cf.append(a[: int(np.nonzero(np.abs(a) > 1e-15)[0].max()) + 1])
        K = max(len(a) for a in cf)
        t0, t1 = psi, (self.H(psi, V, q, ph) - c * psi) / dl
        outs = [complex(a[0]) * t0 + complex(a[1]) * t1 for a in cf]
        for k in range(2, K):
            t0, t1 = t1, (2.0 / dl) * (self.H(t1, V, q, ph) - c * t1) - t0
            outs = [o + complex(a[k]) * t1 if k < len(a) else o for o, a in zip(outs, cf)]
        return outs

    def _all(self, psi, V, A, taus, chunk):
        res = [[] for _ in taus]
        for k in range(psi.shape[0]):
            q = torch.tensor(self.s["kpts"][k], device="cuda") + A
            parts = [self._series(psi[k, i:i + chunk], V, q, taus) for i in range(0, psi.shape[1], chunk)]
            for r, o in zip(res, zip(*parts)):
                r.append(torch.cat(o))
        return [torch.stack(r) for r in res]

    def set_window(self, V, A):
        """An interval that holds the spectrum (any one gives the same exponentials)."""
        v, b = 0.5 * (V[0] + V[1]), 0.5 * ((V[0] - V[1]) ** 2 + V[2] ** 2 + V[3] ** 2).sqrt()
        sums = torch.zeros(self.n ** 3, dtype=torch.float64, device="cuda")
        for idx, _, beta in self.atoms:
            sums[idx] += beta.abs().sum(0)
        gram = max(float((beta.abs() @ sums[idx]).max()) * self.dV for idx, _, beta in self.atoms)
        nl = gram * float(torch.linalg.eigvalsh(self.D).abs().max())
        kin = max(0.5 * sum(float((self.g[a] + self.s["kpts"][k, a] + self.s["A"][j, a]).abs().max()) ** 2 for a in range(3))
                  for k in range(len(self.s["kpts"])) for j in range(2))
        lo, hi = float(v.min() - b.max()) - nl, float(v.max() + b.max()) + nl + kin
        self.window = (lo - 0.03 * (hi - lo), hi + 0.03 * (hi - lo))

    def step(self, psi, A, B, chunk):
        """One ETRS step from t = 0 with the field nodes A[0..1], B[0..1]."""
        V0, _ = self.potential(self.rho(psi), B[0])
        with torch.no_grad():
            self.set_window(V0, A)
        dt = self.s["dt"]
        pred, phi = self._all(psi, V0, A[0], (dt, 0.5 * dt), chunk)
        for _ in range(1 + self.case["n_sc"]):
            V1, _ = self.potential(self.rho(pred), B[1])
            (pred,) = self._all(phi, V1, A[1], (0.5 * dt,), chunk)
        return pred


def exact(case, seed):
    s = system(case, seed)
    if work(case)["flops"] > 1.0e12:  # over 20 s in FP64
        return None
    x = _Exact(case, s)
    if case["do"] == "hartree":
        return x.hartree(_density_input(case, s, seed))
    fp64 = case["precision"] == "fp64"
    psi = spinors(case, s, seed, torch.complex128 if fp64 else torch.complex64).to(torch.complex128)
    A, B = torch.tensor(s["A"][:2], device="cuda"), torch.tensor(s["B"][:2], device="cuda")
    chunk = max(1, int(3e9 / (32.0 * case["n"] ** 3)))
    if case["do"] == "step":
        return x.step(psi, A, B, chunk)
    V, p = x.potential(x.rho(psi), B[0])
    if case["do"] == "apply":
        q = torch.tensor(s["kpts"], device="cuda") + A[0]
        return torch.stack([torch.cat([x.H(psi[k, i:i + chunk], V, q[k], x.phases(q[k])) for i in range(0, psi.shape[1], chunk)])
                            for k in range(len(q))])
    if case["do"] == "gradient":
        A.requires_grad_(True)
        B.requires_grad_(True)
        out = x.step(psi, A, B, psi.shape[1])
        r = x.rho(out)
        loss = (r[0] - r[1]).sum() * x.dV
        loss.backward()
        dA, dB = (np.vstack([g.grad.cpu().numpy(), np.zeros((len(s["t"]) - 2, 3))]) for g in (A, B))
        return dict(loss=float(loss.detach()), dA=dA, dB=dB, psi=out.detach())
    rho, n, m, b = x.rho(psi), p["n"], p["m"], p["b"]
    kin = nl = 0.0
    soc = np.zeros(3)
    for k in range(psi.shape[0]):
        q = torch.tensor(s["kpts"][k], device="cuda") + A[0]
        for i in range(0, psi.shape[1], chunk):
            v, w = psi[k, i:i + chunk], x.wf[k, i:i + chunk]
            kin += float((w * (v.conj() * x.kinetic(v, q)).real.sum((1, 2, 3, 4))).sum()) * x.dV
            for c in x.coefficients(v, x.phases(q)):
                nl += float((w * (c.conj() * (c @ x.D.T)).real.sum(1)).sum())
                soc += [float((w * (c.conj() * (c @ T.T)).real.sum(1)).sum()) for T in x.torque_mats]
    loc, har, exc = (float(v.sum()) * x.dV for v in (x.vloc * n, 0.5 * p["vH"] * n, p["e"]))
    pot = float((rho * torch.stack([p["vbar"] + b[2], p["vbar"] - b[2], 2.0 * b[0], -2.0 * b[1]])).sum()) * x.dV
    M = m.sum((1, 2, 3)) * x.dV
    zee = torch.linalg.cross(B[0], M)
    total = kin + nl + loc + har + exc + 0.5 * float((B[0] * M).sum())
    xs = _grid(s)
    best, owner = torch.full((x.n,) * 3, math.inf, dtype=torch.float64, device="cuda"), torch.zeros((x.n,) * 3, dtype=torch.int64, device="cuda")
    for a, R in enumerate(s["pos"]):
        d = [v - R[ax] for ax, v in enumerate(xs)]
        d = [v - s["L"][ax] * torch.round(v / s["L"][ax]) for ax, v in enumerate(d)]
        d2 = d[0] ** 2 + d[1][:, None] ** 2 + d[2][:, None, None] ** 2
        owner, best = torch.where(d2 < best, a, owner), torch.minimum(best, d2)
    cells = [owner == a for a in range(len(s["pos"]))]
    norms = torch.stack([torch.stack([(v.real ** 2 + v.imag ** 2).sum() for v in psi[k]]) for k in range(psi.shape[0])]) * x.dV
    return dict(n=n, m=m, norms=norms, moments=torch.stack([(m * c).sum((1, 2, 3)) for c in cells]) * x.dV,
                electrons=torch.stack([(n * c).sum() for c in cells]) * x.dV, soc=soc, torque=soc + zee.cpu().numpy(),
                E=[kin, nl, loc, har, exc, total, pot, float(n.sum()) * x.dV], M=M)
