"""The mixed path's residual is formed in FP64 whatever the size of its values: sources in tiny
units leave the FP32 iterate within FP32's normal range, but products of FP32 parts would
not be."""
import numpy as np
import pytest

from _gpu import dev, host, random_problem
from oracle.transport import Discretization, residual_terms

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p", [1, 2, 3, 4])
@pytest.mark.parametrize("log2_scale", [0, -110])
def test_first_residual_keeps_fp64_at_any_scale(lib, p, log2_scale):
    """One fixed pass gives the FP32 sweep's psi; with two, info.rel_residual is ||r|| / ||b||
    there.  r is summed in FP64 over fewer than 2^7 terms per row, so it differs from the oracle's
    r of the same psi by less than 2^7 2^-53 of its terms' size, and so does the norm."""
    from paper_2301_04758_gb300.api import Mesh
    nx, ny, sn = 3, 2, 4
    prob = random_problem(nx, ny, 3, 0.06, p, sn, seed=800 + p)
    scale = 2.0 ** log2_scale
    phi_in, q, inflow = (scale * prob[k] for k in ("phi_in", "source", "inflow"))
    mesh = Mesh(nx, ny, 3, p, 0.06)

    def sweep(passes):
        return mesh.sweep(dev(prob["sigma_t"]), dev(prob["sigma_s"]), prob["omega"], prob["weights"], phi_in=dev(phi_in),
                          source=dev(q), inflow=dev(inflow), precision="mixed", tol=-1.0, max_passes=passes, info=True)
    psi = host(sweep(1)[0])
    assert np.abs(psi).min() > 2.0 ** -126
    disc = Discretization(nx, ny, 3, 0.06, p)
    args = (disc, prob["omega"], prob["sigma_t"], prob["sigma_s"])
    data = dict(phi_in=phi_in, source=q, inflow=inflow)
    r, size = residual_terms(*args, psi, **data)
    b, _ = residual_terms(*args, np.zeros_like(psi), **data)
    r, size, b = r / scale, size / scale, b / scale   # norms of squares within range
    rel = sweep(2)[1]["rel_residual"]
    tol = 2.0 ** -46 * np.linalg.norm(size) / np.linalg.norm(r)
    assert abs(rel / (np.linalg.norm(r) / np.linalg.norm(b)) - 1.0) < tol, (rel, tol)
