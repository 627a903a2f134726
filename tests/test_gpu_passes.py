"""GPU checks of the passes whose work is split by size: the Poisson solve's line tiles, the FFT passes
and the kinetic energy at every grid, the projector gather over one or many CTAs per atom and one or
two spinors per thread, and the tables kept per A(t).  Each against the FP64 oracle (or a plain FFT)
at the sizes where a tile, a chunk or a pair has a remainder."""
import numpy as np
import pytest

from oracle import System
from oracle.tddft import FieldTable
from paper_2506_21908_gb300 import synthetic as S

pytestmark = pytest.mark.gpu


def rel(a, b):
    return float(np.abs(np.asarray(a) - np.asarray(b)).max() / np.abs(np.asarray(b)).max())


# FFT rounding: a few eps per radix step, log2(n^3) <= 18 steps each way, well below 1e-13 of the
# largest value.
@pytest.mark.parametrize("n", [8, 12, 16, 24, 32, 48, 64])
def test_poisson_solve_matches_a_plain_fft(lib, n):
    import torch
    from paper_2506_21908_gb300 import _lib
    L = np.array([7.0, 9.5, 12.25])
    rho = np.random.default_rng(n).uniform(0.0, 1.0, (n, n, n))
    f = np.fft.fftfreq(n) * n * 2.0 * np.pi
    g2 = (f / L[2])[:, None, None] ** 2 + (f / L[1])[:, None] ** 2 + (f / L[0]) ** 2
    c = np.divide(4.0 * np.pi, g2, out=np.zeros_like(g2), where=g2 > 0)
    ref = np.fft.ifftn(np.fft.fftn(rho) * c).real
    d = torch.from_numpy(rho).cuda()
    out = torch.empty_like(d)
    _lib.hartree_noalloc(d, out, L)
    assert rel(out.cpu().numpy(), ref) <= 1e-13
    _lib.hartree_noalloc(d, d, L)  # in place
    assert np.array_equal(d.cpu().numpy(), out.cpu().numpy())


def _system(n, natoms, nstates, nk, lmax=2, seed=3):
    wl = S.small_parity(n=n, natoms=natoms, nstates=nstates, nk=nk, lmax=lmax, seed=seed)
    return wl, S.small_parity_states(wl), System.from_workload(wl)


# (1 atom, 1 spinor): the most CTAs per atom; 40 spinors of 5 atoms: one; odd counts: one spinor per
# thread in FP32, even: two.  FP64 1e-12 and FP32 2e-5 of the largest value, the bounds of the
# Hamiltonian apply at the other sizes.
@pytest.mark.parametrize("precision,tol", [(0, 1e-12), (1, 2e-5)])
@pytest.mark.parametrize("n,natoms,nstates,nk,lmax", [(8, 1, 1, 1, 2), (12, 2, 2, 2, 1), (24, 1, 1, 1, 0), (32, 1, 1, 2, 2),
                                                      (32, 3, 4, 1, 2), (16, 5, 40, 1, 1), (48, 2, 3, 1, 2)])
def test_apply_and_kinetic_energy_at_every_split(lib, precision, tol, n, natoms, nstates, nk, lmax):
    from paper_2506_21908_gb300 import _lib
    wl, psi, s = _system(n, natoms, nstates, nk, lmax)
    A, B = FieldTable(wl.times, wl.A, wl.B).at(wl.dt)
    V, _ = s.potential(s.rho_v(psi), B)
    ref = s.apply_h(psi, V, A)
    h = _lib.TDDFT.from_workload(wl, precision=precision, e_min=-50.0, e_max=600.0)
    h.set_fields(wl.times, wl.A, wl.B)
    h.set_states(psi, wl.dt)
    assert rel(h.apply_hamiltonian(psi), ref) <= tol
    _, _, E, _ = h.observables(fields=False)
    h.close()
    wf = s.kw[:, None] * s.occ
    ekin = sum(wf[k, i] * np.vdot(psi[k, i], s.apply_kinetic(psi[k], s.kpts[k] + A)[i]).real * s.grid.dV
               for k in range(nk) for i in range(nstates))
    assert abs(E["kin"] - ekin) <= (1e-11 if precision == 0 else 5e-6) * abs(ekin)


@pytest.mark.parametrize("precision", [0, 1])
def test_tables_follow_the_field(lib, precision):
    """The phase and kinetic tables belong to one A: a handle that has stepped in one field gives, in
    another, the bits of a fresh handle."""
    from paper_2506_21908_gb300 import _lib
    wl, psi, _ = _system(16, 2, 3, 2)

    def run(h, A):
        h.set_fields(wl.times, A, wl.B)
        h.set_states(psi, 0.0)
        h.step(2)
        E = h.observables(fields=False)[2]
        return h.get_states(), E["kin"], E["nl"]

    h = _lib.TDDFT.from_workload(wl, precision=precision, e_min=-30.0, e_max=250.0)
    first = run(h, wl.A)
    other = run(h, wl.A * 0.5 + 0.1)
    again = run(h, wl.A)
    h.close()
    f = _lib.TDDFT.from_workload(wl, precision=precision, e_min=-30.0, e_max=250.0)
    fresh = run(f, wl.A * 0.5 + 0.1)
    f.close()
    assert np.array_equal(other[0], fresh[0]) and other[1:] == fresh[1:]
    assert np.array_equal(again[0], first[0]) and again[1:] == first[1:]
    assert not np.array_equal(first[0], other[0])


def test_every_call_forms_its_own_tables(lib):
    """A call's launches do not depend on the calls before it."""
    from paper_2506_21908_gb300 import _lib
    wl, psi, _ = _system(16, 2, 3, 1)
    h = _lib.TDDFT.from_workload(wl, precision=0, e_min=-30.0, e_max=250.0)
    h.set_fields(wl.times, wl.A, wl.B)
    h.set_states(psi, 0.0)
    count = [h.info()["launches"]]
    for _ in range(3):
        h.apply_hamiltonian(psi)
        count.append(h.info()["launches"])
    h.close()
    assert len(set(np.diff(count))) == 1


def test_crank_nicolson_order_is_that_of_its_series(lib):
    """|rho| < 1 bounds the coefficients 4 |rho|^k / (beta |sqrt(x0^2 - 1)|): the FP64 order at 1e-16
    follows from the window and the step."""
    from paper_2506_21908_gb300 import _lib
    wl, psi, _ = _system(16, 1, 2, 1)
    lo, hi = -20.0, 120.0
    h = _lib.TDDFT.from_workload(wl, precision=0, exp_kind=2, e_min=lo, e_max=hi)
    h.set_states(psi, 0.0)
    K = h.info()["K_full"]
    h.close()
    x0 = 1j * (1 + 0.25j * wl.dt * (hi + lo)) / (0.25 * wl.dt * (hi - lo))
    sq = np.sqrt(x0 * x0 - 1)
    sq = sq if abs(x0 + sq) > 1 else -sq
    a = 4.0 / (0.25 * wl.dt * (hi - lo)) / abs(sq) * np.abs(x0 + sq) ** -np.arange(400.0)
    assert K == int(np.nonzero(a >= 1e-16)[0].max())


def test_crank_nicolson_with_a_vanishing_step_is_the_identity(lib):
    from paper_2506_21908_gb300 import _lib
    wl, psi, _ = _system(16, 1, 2, 1)
    wl.dt = 1e-200
    h = _lib.TDDFT.from_workload(wl, precision=0, exp_kind=2, e_min=-20.0, e_max=120.0)
    h.set_states(psi, 0.0)
    assert h.info()["K_full"] == 0
    h.step(1)
    out = h.get_states()
    h.close()
    assert rel(out, psi) <= 1e-15


@pytest.mark.parametrize("nstates", [1, 33])
def test_split_bricks_match_the_cuda_core_projectors(lib, nstates):
    """Bricks shared by two CTAs (fewer than 608) and a last component group of two: one step with the
    split FP16 products against the FP32 CUDA-core contraction (both within 2e-5 of the oracle)."""
    from paper_2506_21908_gb300 import _lib
    wl, psi, _ = _system(48, 3, nstates, 1)
    out = []
    for mode in (_lib.PROJ_FP32, _lib.PROJ_F16X3):
        h = _lib.TDDFT.from_workload(wl, precision=1, proj_mode=mode, e_min=-50.0, e_max=500.0)
        h.set_fields(wl.times, wl.A, wl.B)
        h.set_states(psi, 0.0)
        h.step(1)
        h.observables(fields=False)
        out.append(h.get_states())
        h.close()
    assert rel(out[1], out[0]) <= 4e-5
