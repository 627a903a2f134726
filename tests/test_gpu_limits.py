"""GPU checks at the limits of what a handle accepts: spheres that hold no grid point, series of order 0
and vanishing steps, the projector gather's splits that other tests' sizes do not reach, and calls that
follow a refused one.  Against the FP64 oracle or a closed form."""
import numpy as np
import pytest

from oracle import System
from oracle.tddft import FieldTable
from paper_2506_21908_gb300 import synthetic as S

pytestmark = pytest.mark.gpu


def rel(a, b):
    return float(np.abs(np.asarray(a) - np.asarray(b)).max() / np.abs(np.asarray(b)).max())


# FP64 1e-12 and FP32 2e-5 of the largest value: the bounds of the Hamiltonian apply at other systems.
@pytest.mark.parametrize("precision,mode,tol", [(0, 0, 1e-12), (1, 1, 2e-5), (1, 2, 2e-5), (1, 3, 2e-5), (1, 4, 2e-5),
                                                (1, 5, 2e-5)])
def test_spheres_without_a_grid_point(lib, precision, mode, tol):
    """Atoms between the grid points with a radius below their distance: no projector entry anywhere, so
    every projector launch skips all of its blocks."""
    from paper_2506_21908_gb300 import _lib
    wl = S.small_parity(n=16, natoms=2, nstates=3, nk=2)
    psi = S.small_parity_states(wl)
    h0 = wl.L[0] / wl.n
    wl.pos[:] = h0 * (np.array([[3, 5, 9], [12, 1, 6]]) + 0.5)
    wl.r_cut = 0.5 * h0  # the nearest grid points are sqrt(3) / 2 spacings away
    s = System.from_workload(wl)
    A, B = FieldTable(wl.times, wl.A, wl.B).at(0.0)
    V, _ = s.potential(s.rho_v(psi), B)
    ref = s.apply_h(psi, V, A)
    out = {}
    for kind in (0, 1):  # Chebyshev (tensor cores: fused epilogue), Taylor (separate scatter)
        h = _lib.TDDFT.from_workload(wl, precision=precision, proj_mode=mode, exp_kind=kind, e_min=-50.0, e_max=500.0)
        h.set_fields(wl.times, wl.A, wl.B)
        h.set_states(psi, 0.0)
        assert rel(h.apply_hamiltonian(psi), ref) <= tol
        assert np.abs(h.torques()["soc"]).max() == 0.0
        h.step(1)
        E = h.observables(fields=False)[2]
        assert E["nl"] == 0.0
        out[kind] = h.get_states()
        if kind == 0 and precision == 0:
            assert np.isfinite(h.backward(1, np.ones((4, wl.n ** 3)))[1]).all()
        h.close()
    # the same step by the CUDA-core form of the same precision
    h = _lib.TDDFT.from_workload(wl, precision=precision, proj_mode=0 if precision == 0 else 1, e_min=-50.0, e_max=500.0)
    h.set_fields(wl.times, wl.A, wl.B)
    h.set_states(psi, 0.0)
    h.step(1)
    assert rel(out[0], h.get_states()) <= 2 * tol
    h.close()


# The order-0 coefficient is the mean of the exponential (or of the Cayley transform) over the window with
# the Chebyshev weight.  psi takes the half step's coefficient twice; FP32 rounds three times (6e-8 each).
# Orders: the exponential drops |J_1| < tol, the Cayley transform |a_1| < tol, about 2 |J_1|.
@pytest.mark.parametrize("precision,tol", [(0, 1e-14), (1, 4e-7)])
@pytest.mark.parametrize("kind,cheb_tol,orders", [(0, 0.05, (0, 0)), (0, 0.025, (1, 0)), (2, 0.1, (0, 0)), (2, 0.05, (1, 0))])
def test_series_of_order_zero(lib, precision, tol, kind, cheb_tol, orders):
    """Both orders 0, and the half step's alone: the states take the coefficient, the potential and the
    density are those of the states, and nothing of them depends on the fields."""
    from paper_2506_21908_gb300 import _lib
    wl = S.small_parity(n=16, natoms=1, nstates=2, nk=1)
    wl.dt = 1e-3
    psi = S.small_parity_states(wl)
    lo, hi = -20.0, 120.0
    E = 0.5 * (lo + hi) + 0.5 * (hi - lo) * np.cos(np.pi * (np.arange(64) + 0.5) / 64)
    tau = 0.5 * wl.dt
    f = np.exp(-1j * tau * E) if kind == 0 else (1 - 0.5j * tau * E) / (1 + 0.5j * tau * E)
    cf = f.mean()
    h = _lib.TDDFT.from_workload(wl, precision=precision, exp_kind=kind, cheb_tol=cheb_tol, e_min=lo, e_max=hi)
    h.set_fields(wl.times, wl.A, wl.B)
    h.set_states(psi, 0.0)
    assert (h.info()["K_full"], h.info()["K_half"]) == orders
    h.step(1)
    n, m, _, norms = h.observables()
    assert rel(h.get_states(), cf * cf * psi) <= tol
    assert np.abs(norms - abs(cf) ** 4).max() <= 2 * tol
    s = System.from_workload(wl)
    V, _ = s.potential(s.rho_v(cf * cf * psi), FieldTable(wl.times, wl.A, wl.B).at(wl.dt)[1])
    assert rel(h.get_potential(), V) <= 4 * tol + 1e-12
    h.set_states(psi, 0.0)
    _, dA, dB = h.backward(1, np.random.default_rng(1).normal(size=(4, wl.n ** 3)))
    assert not dA.any() and not dB.any()
    h.close()


# Every coefficient but the first vanishes and that one is 1: no rounding but the density's own.
@pytest.mark.parametrize("kind", [0, 2])
@pytest.mark.parametrize("dt", [1e-60, -1e-200, 1e-310])
@pytest.mark.parametrize("order", [0, 1, 4])
def test_a_vanishing_step_is_the_identity(lib, kind, dt, order):
    from paper_2506_21908_gb300 import _lib
    wl = S.small_parity(n=16, natoms=1, nstates=2, nk=1)
    wl.dt = dt
    psi = S.small_parity_states(wl)
    h = _lib.TDDFT.from_workload(wl, precision=0, exp_kind=kind, exp_order=order, e_min=-20.0, e_max=120.0)
    h.set_states(psi, 0.0)
    info = h.info()
    assert (info["K_full"], info["K_half"]) == (order, order)
    V = h.get_potential()
    h.step(1)
    norms = h.observables(fields=False)[3]
    assert rel(h.get_states(), psi) <= 1e-15
    assert rel(h.get_potential(), V) <= 1e-14
    assert np.abs(norms - 1.0).max() <= 1e-12
    h.close()


def test_tensor_core_handle_holds_no_gather_workspace(lib):
    """The phases of the CUDA-core gather (16 bytes per entry and k-point) serve a tensor-core handle in
    backward alone: creation takes no more per k-point than its spinor arrays and partial
    products, backward gives back what it took, and its gradient tracks FP64 within the 1e-3 of the
    FP32 path."""
    import torch
    from paper_2506_21908_gb300 import _lib
    free = lambda: torch.cuda.mem_get_info()[0]  # noqa: E731
    n, natoms, nk = 48, 8, 16
    took = {}
    for k in (1, nk):
        wl = S.small_parity(n=n, natoms=natoms, nstates=1, nk=k, lmax=0)
        torch.cuda.synchronize()
        before = free()
        h = _lib.TDDFT.from_workload(wl, precision=1, proj_mode=_lib.PROJ_F16X3, e_min=-20.0, e_max=300.0)
        took[k] = before - free()
        h.close()
    entries = natoms * 4.0 / 3.0 * np.pi * (wl.r_cut * n / wl.L[0]) ** 3
    phases = (nk - 1) * 16 * entries
    arrays = (nk - 1) * 2 * n ** 3 * (7 * 8 + 16)  # seven of spinors and the staging of host states
    arrays += 11 * 4 * n ** 3 * 8  # the band groups of the density at 16 spinors
    partials = (nk - 1) * 2 * natoms * 108 * 512  # at most two images of an atom in each of the 108 bricks
    assert took[nk] - took[1] <= arrays + partials + 0.5 * phases
    wl = S.small_parity(n=16, natoms=2, nstates=2, nk=2)
    wl.dt = 0.02
    psi = S.small_parity_states(wl)
    seed = np.zeros((4, wl.n ** 3))
    seed[0], seed[1] = 1.0, -1.0
    grad = []
    for precision, mode in ((0, 0), (1, _lib.PROJ_F16X3)):
        h = _lib.TDDFT.from_workload(wl, precision=precision, proj_mode=mode, e_min=-30.0, e_max=250.0)
        h.set_fields(wl.times, wl.A, wl.B)
        for _ in range(2):
            h.set_states(psi, 0.0)
            before = free()
            grad.append(h.backward(2, seed)[1:])
            assert free() >= before
        h.step(1)  # the handle steps on as before
        assert h.observables(fields=False)[2]["status"] == 0
        h.close()
    for a, b in ((grad[1], grad[0]), (grad[3], grad[2])):
        assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
    for a, b in zip(grad[2], grad[0]):
        assert np.abs(a - b).max() <= 1e-3 * np.abs(b).max()


def test_a_refused_allocation_is_not_met_again(lib):
    """A handle beyond the device's memory is refused with TDDFT_ERR_OOM; the next one is created and steps
    as if nothing had been asked (the runtime keeps an error until it is read)."""
    from paper_2506_21908_gb300 import _lib
    big = S.small_parity(n=96, natoms=0, nstates=32767, nk=1)  # one spinor array: 927 GB
    wl = S.small_parity(n=16, natoms=2, nstates=2, nk=1)
    psi = S.small_parity_states(wl)
    for _ in range(2):
        with pytest.raises(_lib.TddftError) as e:
            _lib.TDDFT.from_workload(big, precision=0)
        assert e.value.status == -3
        h = _lib.TDDFT.from_workload(wl, precision=0, e_min=-30.0, e_max=250.0)
        h.set_states(psi, 0.0)
        h.step(1)
        assert h.observables(fields=False)[2]["status"] == 0
        h.close()


# The gather's CTAs per atom (proj_chunks): one with two spinors per thread (about 190 entries per atom, no
# partial sums), and the FP32 rule for more than 608 groups of an atom and a spinor pair (16 x 40 with
# 12000 entries each: four).
@pytest.mark.parametrize("precision,tol", [(0, 1e-12), (1, 2e-5)])
@pytest.mark.parametrize("n,natoms,nstates", [(8, 1, 2), (8, 3, 4), (32, 16, 80)])
def test_gather_splits(lib, precision, tol, n, natoms, nstates):
    from paper_2506_21908_gb300 import _lib
    wl = S.small_parity(n=n, natoms=natoms, nstates=nstates, nk=1, lmax=1)
    psi = S.small_parity_states(wl)
    s = System.from_workload(wl)
    A, B = FieldTable(wl.times, wl.A, wl.B).at(wl.dt)
    V, _ = s.potential(s.rho_v(psi), B)
    ref = s.apply_h(psi, V, A)
    h = _lib.TDDFT.from_workload(wl, precision=precision, e_min=-200.0, e_max=600.0)
    h.set_fields(wl.times, wl.A, wl.B)
    h.set_states(psi, wl.dt)
    assert rel(h.apply_hamiltonian(psi), ref) <= tol
    h.close()
