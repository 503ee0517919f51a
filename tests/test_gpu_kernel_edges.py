"""Edges of the dispatch of the element factorisation, the mixed path's first residual and the
hybridized VEF solve: remainders of the tasks per warp and the elements per CTA, boundary
data, pivot fallbacks, tiles wider than a CTA."""
import numpy as np
import pytest

from _gpu import dev, host, rel, random_problem
from oracle.transport import Discretization, sweep as o_sweep, residual_terms

pytestmark = pytest.mark.gpu


def _sweep(prob, **kw):
    from paper_2301_04758_gb300.api import Mesh
    mesh = Mesh(prob["nx"], prob["ny"], prob["m"], prob["p"], prob["alpha"])
    opt = lambda a: None if a is None else dev(a)
    return mesh.sweep(dev(prob["sigma_t"]), dev(prob["sigma_s"]), prob["omega"], prob["weights"],
                      phi_in=opt(prob["phi_in"]), source=dev(prob["source"]), inflow=opt(prob["inflow"]),
                      info=True, **kw)


def _subset(prob, D):
    out = dict(prob, omega=np.ascontiguousarray(prob["omega"][:D]), weights=np.ascontiguousarray(prob["weights"][:D]))
    for k in ("source", "inflow"):
        if out[k] is not None and out[k].ndim == 3:
            out[k] = np.ascontiguousarray(out[k][:D])
    return out


@pytest.mark.parametrize("p", [3, 4])
@pytest.mark.parametrize("nx,ny,sn,D", [(1, 1, 4, 12), (3, 1, 4, 1), (5, 3, 4, 3), (3, 3, 6, 24), (7, 5, 8, 40)])
def test_factorisation_with_partial_warps_and_ctas(lib, p, nx, ny, sn, D):
    """An odd number of elements (the last CTA holds one), direction counts that leave part of a
    warp without tasks, all quadrants in one warp: FP64 within 1e-12 and mixed within 1e-10."""
    prob = _subset(random_problem(nx, ny, 3, 0.06, p, sn, seed=700 + p, aniso=True), D)
    disc = Discretization(nx, ny, 3, 0.06, p)
    ref = o_sweep(disc, prob["omega"], prob["weights"], prob["sigma_t"], prob["sigma_s"], phi_in=prob["phi_in"],
                  source=prob["source"], inflow=prob["inflow"])
    psi, info = _sweep(prob)
    assert rel(host(psi), ref) < 1e-12, info
    psi, info = _sweep(prob, precision="mixed")
    assert rel(host(psi), ref) < 1e-10, info


@pytest.mark.parametrize("p", [1, 2, 3, 4])
@pytest.mark.parametrize("aniso,inflow", [(False, False), (True, True)])
def test_first_residual_of_the_mixed_path(lib, p, aniso, inflow):
    """With one fixed pass psi is the FP32 sweep's result; with two, info.rel_residual is
    ||r|| / ||b|| at that iterate.  The library forms r to about 2^-46 of the terms it sums
    (FP32 pairs) or better, so the ratio agrees with the oracle's element-by-element residual of
    the same psi to 2^-44 of the size of its terms."""
    nx, ny, sn = 9, 7, 6
    prob = random_problem(nx, ny, 3, 0.08, p, sn, seed=720 + p, aniso=aniso, with_inflow=inflow)
    disc = Discretization(nx, ny, 3, 0.08, p)
    args = (disc, prob["omega"], prob["sigma_t"], prob["sigma_s"])
    data = dict(phi_in=prob["phi_in"], source=prob["source"], inflow=prob["inflow"])
    psi0, _ = _sweep(prob, precision="mixed", tol=-1.0, max_passes=1)
    psi0 = host(psi0)
    assert np.array_equal(psi0, psi0.astype(np.float32).astype(np.float64))
    r, size = residual_terms(*args, psi0, **data)
    b, _ = residual_terms(*args, np.zeros_like(psi0), **data)
    _, info = _sweep(prob, precision="mixed", tol=-1.0, max_passes=2)
    tol = 2.0 ** -44 * np.linalg.norm(size) / np.linalg.norm(r)
    assert abs(info["rel_residual"] / (np.linalg.norm(r) / np.linalg.norm(b)) - 1.0) < tol, (info, tol)


def _vef_case(nx, ny, p, seed):
    from test_gpu_hrt import _vef_inputs
    disc = Discretization(nx, ny, 3, 0.05, p)
    return disc, list(_vef_inputs(disc, seed))


@pytest.mark.parametrize("nx,ny,p,tol", [(121, 33, 3, 1e-9), (45, 1, 2, 1e-9), (2, 1, 4, 1e-9)])
def test_hrt_tiles(lib, nx, ny, p, tol):
    """Tiles with more multipliers than half a CTA's threads (11 x 3 elements at p = 3), a mesh
    one element high (no horizontal faces) and a single face, against the direct solution."""
    from paper_2301_04758_gb300.api import Mesh
    from test_gpu_hrt import _oracle
    disc, v = _vef_case(nx, ny, p, 740)
    ref = _oracle(disc, *v)
    phi, P, Eb, Jin, Q0, Q1, st, ss = v
    mesh = Mesh(nx, ny, 3, p, 0.05)
    gphi, gJ, glam, info = mesh.hrt_solve(dev(st), dev(ss), dev(phi), dev(P), dev(Eb), dev(Jin), dev(Q0), dev(Q1),
                                          tol=1e-13)
    assert rel(host(glam), ref["lam"]) < tol, info
    assert rel(host(gphi), ref["phi"]) < tol, info
    assert rel(host(gJ), ref["J"]) < tol, info


@pytest.mark.parametrize("p", [1, 2, 3, 4])
def test_hrt_small_diagonal_pivots(lib, p):
    """Elements with sigma_t = 1e-9: the mass block's pivots fall below 2^-26 of their rows'
    largest entries (the Piola gradient's), so these elements take the partial-pivoting
    inversion.  Their systems have a condition of about 1e9 / h, so phi is compared to 1e-5."""
    from paper_2301_04758_gb300.api import Mesh
    from test_gpu_hrt import _oracle
    disc, v = _vef_case(5, 4, p, 760 + p)
    thin = np.arange(20) % 3 == 0
    v[6] = np.where(thin, 1e-9, v[6])
    v[7] = np.where(thin, 0.5e-9, v[7])
    ref = _oracle(disc, *v)
    phi, P, Eb, Jin, Q0, Q1, st, ss = v
    mesh = Mesh(5, 4, 3, p, 0.05)
    gphi, _, _, info = mesh.hrt_solve(dev(st), dev(ss), dev(phi), dev(P), dev(Eb), dev(Jin), dev(Q0), dev(Q1),
                                      tol=1e-12, max_iter=5000)
    assert rel(host(gphi), ref["phi"]) < 1e-5, info
