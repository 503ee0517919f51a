"""Meshes of different sizes used from several threads at once, each with its own mesh and
stream: a call's launch limits do not depend on what other threads' calls need."""
import threading

import pytest
import torch

from _gpu import dev, random_problem
from _hrt_exact import exact_problem

pytestmark = pytest.mark.gpu


def _hrt_call(n):
    from paper_2301_04758_gb300.api import Mesh
    v = exact_problem(n, n, 1, 850)
    mesh = Mesh(n, n, 1, 1, 0.0)
    args = [dev(v[k]) for k in ("sigma_t", "sigma_s", "phi_tr", "P_tr", "Eb", "Jin", "Q0", "Q1")]
    return lambda: mesh.hrt_solve(*args, tol=1e-14, max_iter=2, check=False)[2]


def _sweep_call(n):
    from paper_2301_04758_gb300.api import Mesh
    prob = random_problem(n, n, 3, 0.1, 1, 4, seed=851)
    mesh = Mesh(n, n, 3, 1, 0.1)
    args = [dev(prob["sigma_t"]), dev(prob["sigma_s"]), prob["omega"], prob["weights"]]
    kw = dict(phi_in=dev(prob["phi_in"]), source=dev(prob["source"]), inflow=dev(prob["inflow"]), apply="separate")
    return lambda: mesh.sweep(*args, **kw)


@pytest.mark.parametrize("call,large,small", [(_hrt_call, 420, 3), (_sweep_call, 160, 4)], ids=["hrt", "sweep"])
def test_small_calls_do_not_disturb_a_large_one(lib, call, large, small):
    """Six threads repeat a small call while one repeats a large one, whose kernels need more
    shared memory: every call succeeds and every result of the large one is the same."""
    big = call(large)
    ref = big().clone()
    errors, stop = [], threading.Event()

    def work(fn, count):
        try:
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream):
                while not stop.is_set() and (count is None or count > 0):
                    out = fn()
                    stream.synchronize()
                    if count is not None:
                        count -= 1
                        assert torch.equal(out, ref)
        except Exception as e:   # reported by the main thread
            errors.append(e)
            stop.set()
    smalls = [call(small) for _ in range(6)]
    torch.cuda.synchronize()
    threads = [threading.Thread(target=work, args=(f, None)) for f in smalls]
    main = threading.Thread(target=work, args=(big, 60))
    for t in threads + [main]:
        t.start()
    main.join()
    stop.set()
    for t in threads:
        t.join()
    assert not errors, errors[0]
