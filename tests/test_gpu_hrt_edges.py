"""Edges of the hybridized VEF solve: thin elements whose inversion needs pivoting, dot products
near the end of FP64's range, status bits after a solve that fails, bounded grid barriers, and
meshes whose Krylov tiles are cut, empty or several to a CTA."""
import time

import numpy as np
import pytest

from _gpu import dev, host, rel, random_problem
from _hrt_exact import exact_problem
from oracle.hrt import HRT
from oracle.transport import Discretization, sweep as o_sweep

pytestmark = pytest.mark.gpu


def _solve(mesh, v, **kw):
    phi, J, lam, info = mesh.hrt_solve(dev(v["sigma_t"]), dev(v["sigma_s"]), dev(v["phi_tr"]), dev(v["P_tr"]),
                                       dev(v["Eb"]), dev(v["Jin"]), dev(v["Q0"]), dev(v["Q1"]), **kw)
    return host(phi), host(J), host(lam), info


@pytest.mark.parametrize("p", [1, 2, 3, 4])
@pytest.mark.parametrize("sigma_t", [1e-7, 1e-3])
def test_thin_element_keeps_the_digits_of_phi(lib, p, sigma_t):
    """One optically thin element: A's pivots are small against G's entries and an elimination
    that takes them all the same loses log10(1 / sigma_t) digits of phi.  Relative changes of
    2^-52 in the entries of the local system move phi by less than 2^-51, so with at most 85
    elimination steps of a few roundings each phi agrees to 85 x 8 x 2^-53 < 1e-13 with the
    system's solution in 50 digits."""
    import mpmath as mp
    from paper_2301_04758_gb300.api import Mesh
    disc = Discretization(1, 1, 3, 0.05, p)
    h, nq = HRT(disc), disc.nq
    one = np.ones((1, disc.n))
    v = dict(sigma_t=np.full(1, sigma_t), sigma_s=np.full(1, 0.9 * sigma_t), phi_tr=one,
             P_tr=np.stack([one / 3, 0 * one, one / 3]), Eb=np.full((4, nq), 0.5), Jin=np.full((4, nq), -0.1),
             Q0=one, Q1=np.zeros((2, 1, disc.n)))
    Eq, Ef = h.eddington_data(v["phi_tr"], v["P_tr"])
    L, _, _, g, f = h.element(0, v["sigma_t"], v["sigma_t"] - v["sigma_s"], Eq, Ef, v["Eb"], v["Jin"],
                              np.ones((1, nq * nq)))
    with mp.workdps(50):
        x = mp.lu_solve(mp.matrix(L.tolist()), mp.matrix(np.concatenate([g, f]).tolist()))
    ref = np.array([float(t) for t in x])[h.nJ:]
    phi = _solve(Mesh(1, 1, 3, p, 0.05), v)[0]
    assert rel(phi[0], ref) < 1e-13


@pytest.mark.parametrize("kind", ["nan_moment", "pending_timeout"])
def test_a_failed_solve_leaves_no_status_behind(lib, kind):
    """A solve that ends without converging reports what its kernels recorded (a wait that ran
    out before the missing convergence) and leaves the mesh clean: the next sweep and the next
    solve succeed."""
    from paper_2301_04758_gb300 import _lib
    from paper_2301_04758_gb300.api import Mesh
    nx, ny, p = 6, 5, 2
    v = exact_problem(nx, ny, p, 830)
    prob = random_problem(nx, ny, 1, 0.0, p, 4, seed=831)
    mesh = Mesh(nx, ny, 1, p, 0.0)
    bad, kw, want = dict(v), dict(tol=1e-13), _lib.VEF_ERR_NOT_CONVERGED
    if kind == "nan_moment":
        bad["phi_tr"] = v["phi_tr"].copy()
        bad["phi_tr"][7, 0] = np.nan
    else:
        kw, want = dict(tol=1e-13, max_iter=1), _lib.VEF_ERR_TIMEOUT
        assert lib.vef_mesh_inject_status(mesh.handle, _lib.VEF_STATUS_TIMEOUT, None) == _lib.VEF_OK
    with pytest.raises(_lib.VefError) as err:
        _solve(mesh, bad, **kw)
    assert err.value.status == want, err.value
    psi, info = mesh.sweep(dev(prob["sigma_t"]), dev(prob["sigma_s"]), prob["omega"], prob["weights"],
                           phi_in=dev(prob["phi_in"]), source=dev(prob["source"]), inflow=dev(prob["inflow"]), info=True)
    ref = o_sweep(Discretization(nx, ny, 1, 0.0, p), prob["omega"], prob["weights"], prob["sigma_t"], prob["sigma_s"],
                  phi_in=prob["phi_in"], source=prob["source"], inflow=prob["inflow"])
    assert rel(host(psi), ref) < 1e-12 and info["timed_out"] == 0
    phi, J, lam, _ = _solve(mesh, v, tol=1e-13)
    assert rel(phi, v["phi"]) < 1e-10 and rel(J, v["J"]) < 1e-10 and rel(lam, v["lam"]) < 1e-10


def test_dot_products_near_the_end_of_the_range(lib):
    """Sources scaled until ||r||^2 = 2^1021.7: the first iteration divides by r_hat . v between
    2^1022 and 2^1024, whose reciprocal is below FP64's normal range.  The problem is linear, so
    the solution scales with the sources."""
    from paper_2301_04758_gb300.api import Mesh
    p = 2
    v = exact_problem(2, 1, p, 840)
    disc = Discretization(2, 1, 1, 0.0, p)
    h = HRT(disc)
    ref = h.solve(v["sigma_t"], v["sigma_s"], *h.eddington_data(v["phi_tr"], v["P_tr"]), v["Eb"], v["Jin"],
                  np.einsum("qj,ej->eq", disc.B, v["Q0"]), np.einsum("qj,cej->eqc", disc.B, v["Q1"]))
    scale = 2.0 ** 510.85 / np.linalg.norm(ref["r"])
    big = dict(v, Jin=scale * v["Jin"], Q0=scale * v["Q0"], Q1=scale * v["Q1"])
    phi, J, lam, info = _solve(Mesh(2, 1, 1, p, 0.0), big, tol=1e-13)
    for got, key in ((phi, "phi"), (J, "J"), (lam, "lam")):
        assert rel(got / scale, v[key]) < 1e-11, info


def test_grid_barrier_gives_up(lib):
    """The grid barrier's wait runs out when an arrival is missing, with the status for it, and a
    solve that begins with a timeout pending leaves at its first barriers, says so and lets the
    next one succeed."""
    from paper_2301_04758_gb300 import _lib
    from paper_2301_04758_gb300.api import Mesh
    polls = 1 << 12
    assert lib.vef_grid_wait_selftest(1, polls, None) == _lib.VEF_OK
    t = time.perf_counter()
    st = lib.vef_grid_wait_selftest(0, polls, None)
    elapsed = time.perf_counter() - t
    print(f"{polls} polls ran out in {elapsed * 1e3:.2f} ms ({elapsed / polls * 1e9:.0f} ns per poll, launch included)")
    assert st == _lib.VEF_ERR_TIMEOUT and elapsed < 5.0
    assert lib.vef_grid_wait_selftest(0, 0, None) == _lib.VEF_ERR_INVALID_ARG
    assert lib.vef_grid_wait_selftest(0, (1 << 24) + 1, None) == _lib.VEF_ERR_INVALID_ARG
    n, p = 48, 2
    v = exact_problem(n, n, p, 860)
    mesh = Mesh(n, n, 1, p, 0.0)
    _solve(mesh, v, tol=1e-13)
    assert lib.vef_mesh_inject_status(mesh.handle, _lib.VEF_STATUS_TIMEOUT, None) == _lib.VEF_OK
    t = time.perf_counter()
    with pytest.raises(_lib.VefError, match="grid barrier") as err:
        _solve(mesh, v, tol=1e-13)
    assert err.value.status == _lib.VEF_ERR_TIMEOUT and time.perf_counter() - t < 0.5
    phi, J, lam, _ = _solve(mesh, v, tol=1e-13)
    assert rel(phi, v["phi"]) < 1e-9 and rel(J, v["J"]) < 1e-9 and rel(lam, v["lam"]) < 1e-9


@pytest.mark.parametrize("nx,ny,p,least", [(1090, 1, 2, 0), (1, 1090, 3, 0), (500, 5, 1, 0), (12600, 7, 2, 0), (7, 7500, 4, 0),
                                           (640, 640, 2, 257)],
                         ids=["cut_with_empty", "cut_upright", "cut_cells", "tiles_per_cta", "tiles_per_cta_upright",
                              "cut_square_two_launches"])
def test_krylov_tiles_of_large_and_long_meshes(lib, nx, ny, p, least):
    """Cells of the coarse grid cut into several tiles: because a strip has few cells (at 1090
    the last cell's last tile is empty), because the staged vector would not fit (then more tiles
    than CTAs, each taking its share), and more iterations than one launch runs.  phi, J and the
    multipliers against the exact solution; absorption keeps H's condition below about 1e3 per
    coarse cell, so a relative residual of 1e-12 leaves 1e-9."""
    from paper_2301_04758_gb300.api import Mesh
    scale = max(nx, ny) / 10 if min(nx, ny) < 100 else 1.0
    v = exact_problem(nx, ny, p, 870, sigma=(0.5 * scale, 5.0 * scale))
    phi, J, lam, info = _solve(Mesh(nx, ny, 1, p, 0.0), v, tol=1e-12)
    assert info["iterations"] >= least and info["multipliers"] == lam.size, info
    assert rel(phi, v["phi"]) < 1e-9 and rel(J, v["J"]) < 1e-9 and rel(lam, v["lam"]) < 1e-9, info


def test_a_strip_keeps_the_device_busy(lib):
    """An iteration on 10000 x 1 elements takes less than twice one on 100 x 100 (3.7 times when
    each of the strip's eleven coarse cells was one CTA's)."""
    from paper_2301_04758_gb300.api import Mesh
    import torch

    def per_iteration(nx, ny):
        scale = max(nx, ny) / 10
        v = exact_problem(nx, ny, 2, 880, sigma=(0.5 * scale, 5.0 * scale))
        mesh = Mesh(nx, ny, 1, 2, 0.0)
        args = [dev(v[k]) for k in ("sigma_t", "sigma_s", "phi_tr", "P_tr", "Eb", "Jin", "Q0", "Q1")]

        def run(its):
            times = []
            for _ in range(7):
                torch.cuda.synchronize()
                t = time.perf_counter()
                info = mesh.hrt_solve(*args, tol=1e-15, max_iter=its, check=False)[3]
                times.append(time.perf_counter() - t)
                assert info["iterations"] == its
            return sorted(times)[3]
        return (run(34) - run(4)) / 30
    strip, square = per_iteration(10000, 1), per_iteration(100, 100)
    print(f"strip {strip * 1e6:.1f} us, square {square * 1e6:.1f} us per iteration")
    assert strip < 2.0 * square


# pairs of sizes and two seeds each: errors of single solves scatter by a factor of ten
_SIZES = [(13, 17), (19, 23), (26, 31), (40, 40), (33, 29), (45, 37), (22, 41), (51, 14), (28, 28), (37, 43), (16, 16),
          (32, 32), (24, 36), (30, 50)]


def _mean_error(key, sigma, scatter, p=1):
    """Geometric mean over the sizes of the relative error of phi or J, iterated until the
    residual no longer falls."""
    from paper_2301_04758_gb300.api import Mesh
    errors = []
    for nx, ny in _SIZES:
        for seed in (100, 101):
            v = exact_problem(nx, ny, p, seed, sigma, scatter)
            phi, J, _, _ = _solve(Mesh(nx, ny, 1, p, 0.0), v, tol=1e-15, max_iter=400, check=False)
            errors.append(rel({"phi": phi, "J": J}[key], v[key]))
    return np.exp(np.mean(np.log(errors)))


@pytest.mark.parametrize("sigma,scatter,limit", [((1e-3, 1e-2), (0.5, 0.9), 4.6e-11), ((0.5, 5.0), (0.3, 0.95), 8.4e-14),
                                                 ((0.5, 5.0), (1.0, 1.0), 8.2e-14)], ids=["thin", "mid", "scattering"])
def test_the_multiplier_update_rounds_once(lib, sigma, scatter, limit):
    """J's mean error against the exact solution stays within an eighth of what it is with one
    rounding at the size of lambda per iteration (4.1e-11, 7.5e-14, 7.3e-14; with two, by a
    chain of multiply-adds, 5.1e-11, 9.2e-14, 9.4e-14)."""
    assert _mean_error("J", sigma, scatter) < limit


@pytest.mark.parametrize("sigma,scatter,limit", [((1e-3, 1e-2), (0.5, 0.9), 3.4e-12), ((0.5, 5.0), (0.3, 0.95), 1.1e-14),
                                                 ((0.5, 5.0), (1.0, 1.0), 1.8e-14)], ids=["thin", "mid", "scattering"])
def test_reference_tables_keep_the_element_balance(lib, sigma, scatter, limit):
    """phi's mean error against the exact solution stays within a fifth of what the reference
    divergences and face fluxes, summed term by term over the points, gave (2.8e-12, 9.2e-15,
    1.5e-14): their rounding breaks every element's balance alike, so in thin and scattering
    media phi collects it (8.6e-12, 1.4e-14, 2.6e-14 with products formed in another order)."""
    assert _mean_error("phi", sigma, scatter) < limit
