"""A VEF problem on a straight uniform mesh of the unit square whose discrete solution is known
in closed form: E = I / 3, polynomial scalar flux and current that the discrete spaces hold, and
per-element cross sections, with the sources and boundary data that go with them.  Works at any
mesh size, since nothing is assembled."""
import numpy as np

from oracle.basis import gll_points, gauss_legendre


def exact_problem(nx, ny, p, seed, sigma=(0.5, 5.0), scatter=(0.3, 0.95)):
    """dict of the inputs of Mesh.hrt_solve (numpy) and the exact phi [E][n], J [E][nJ] and
    lam [faces][p+1]."""
    rng = np.random.default_rng(seed)
    E, q = nx * ny, p + 1
    hx, hy = 1.0 / nx, 1.0 / ny
    c = rng.uniform(-0.2, 0.2, 12)
    k2 = 1.0 if p >= 2 else 0.0

    def phi(x, y):
        return 1.0 + c[0] * x + c[1] * y + c[2] * x * y + k2 * (c[3] * x * x + c[4] * y * y)

    def jx(x, y):
        return c[5] + c[6] * x + c[7] * y + c[8] * x * y

    def jy(x, y):
        return c[9] + c[10] * x + c[11] * y - c[6] * x * y

    st = rng.uniform(*sigma, E)
    ss = rng.uniform(*scatter, E) * st
    i, j = np.tile(np.arange(nx), ny), np.repeat(np.arange(ny), nx)
    nd, g, cl = gll_points(p), gauss_legendre(p + 1)[0], gll_points(p + 1)
    s = gauss_legendre(p + 2)[0]

    def at(rx, ry):   # coordinates of reference points (rx fastest) in every element
        return ((i[:, None] + np.tile(rx, len(ry))[None]) * hx, (j[:, None] + np.repeat(ry, len(rx))[None]) * hy)
    x, y = at(nd, nd)
    gx, gy = c[0] + c[2] * y + 2 * k2 * c[3] * x, c[1] + c[2] * x + 2 * k2 * c[4] * y
    div = c[6] + c[8] * y + c[11] - c[6] * x
    Q0 = div + (st - ss)[:, None] * phi(x, y)
    Q1 = np.stack([st[:, None] * jx(x, y) + gx / 3.0, st[:, None] * jy(x, y) + gy / 3.0])
    J = np.concatenate([hy * jx(*at(cl, g)), hx * jy(*at(g, cl))], axis=1)
    # boundary faces: bottom, right, top, left
    tx, ty = (np.arange(nx)[:, None] + s) * hx, (np.arange(ny)[:, None] + s) * hy
    zx, zy = np.zeros_like(tx), np.zeros_like(ty)
    Eb = 0.5
    Jin = np.concatenate([(-jy(tx, zx) - Eb * phi(tx, zx)) / 2, (jx(zy + 1, ty) - Eb * phi(zy + 1, ty)) / 2,
                          (jy(tx, zx + 1) - Eb * phi(tx, zx + 1)) / 2, (-jx(zy, ty) - Eb * phi(zy, ty)) / 2])
    # interior faces: vertical j (nx - 1) + i, then horizontal
    vi, vj = np.tile(np.arange(1, nx), ny), np.repeat(np.arange(ny), nx - 1)
    hi, hj = np.tile(np.arange(nx), ny - 1), np.repeat(np.arange(1, ny), nx)
    lam = np.concatenate([phi(vi[:, None] * hx + 0 * g, (vj[:, None] + g) * hy),
                          phi((hi[:, None] + g) * hx, hj[:, None] * hy + 0 * g)])
    one = np.ones((E, q * q))
    return dict(sigma_t=st, sigma_s=ss, phi_tr=one, P_tr=np.stack([one / 3, 0 * one, one / 3]),
                Eb=np.full(Jin.shape, Eb), Jin=Jin, Q0=Q0, Q1=Q1, phi=phi(x, y), J=J, lam=lam)
