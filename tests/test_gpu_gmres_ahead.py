"""FP64 GMRES with iterations launched ahead of the host's Givens update: the
guesses must not show in the results.

A solve cut off after k iterations (odd and even k: the dot products of
consecutive iterations use two buffers), with short and long cycles and with
the second Gram-Schmidt pass, reports exactly the first k residuals of the
uncut one -- the kernels and their order are the same, so the comparison is
of bits.  The last estimate of a cycle equals the true residual up to the
loss of orthogonality: 1e-6 relative while it is above 1e-9.  A loose
tolerance stops where a tight one passed it."""
import numpy as np
import pytest

from gpu_cases import dev, host, rel

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def case(cuda_device):
    from oracle import mac, schur
    from paper_2501_15314_gb300 import workloads as wl
    from paper_2501_15314_gb300.api import IBMSolver
    W = wl.config(1)
    g = mac.Grid(W.n)
    sysm = schur.SchurSystem(g, W.X)
    rng = np.random.default_rng(23)
    u = rng.standard_normal(g.n_faces) * g.interior_face_mask_packed()
    b = sysm.rhs_scalar(mac.apply_GT(g, u), rng.standard_normal(sysm.k))
    ref, _, _, _ = schur.solve_schur(sysm, b, rtol=1e-13)
    s = IBMSolver(W.n, Re=W.Re, dt=W.dt)
    s.set_markers(dev(W.X))
    yield s, dev(b), ref
    s.close()


@pytest.mark.parametrize("restart,reorth", [(3, 0), (4, 1), (30, 0), (30, 1)])
def test_cut_off_solves_are_prefixes(case, restart, reorth):
    s, b, ref = case
    kw = dict(precond_prec=0, arnoldi=0, rtol=1e-13, restart=restart, reorth=reorth)
    p, st = s.solve_schur(b, maxit=400, **kw)
    assert rel(host(p), ref) < 1e-10
    hist, n = st["relres_hist"], st["iters"]
    for k in (1, 2, 3, 4, 5, n - 1):
        _, cut = s.solve_schur(b, maxit=k, raise_on_error=False, **kw)
        assert cut["status"] != 0 and cut["iters"] == k
        assert cut["relres_hist"] == hist[:k]
        if hist[k - 1] > 1e-9:
            assert abs(cut["relres_true"] / hist[k - 1] - 1.0) < 1e-6
    for k in (2, 3):
        _, cut = s.solve_schur(b, maxit=400, **{**kw, "rtol": 1.0001 * hist[k]})
        assert cut["iters"] == k + 1 and cut["relres_hist"] == hist[:k + 1]
