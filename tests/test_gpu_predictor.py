"""The momentum predictor where its red-black layout has its edges: odd and
even x-extents, rows of less than one, of several and of one and a part of the
thread groups of 8, 16 and 32, one plane per thread and many, and viscous
numbers from nearly none to large (one to many half-steps per correction).
Whole steps without markers against the oracle's, every term of Eq. (ustar)
active; tolerance 1e-10, the repository's parity."""
import numpy as np
import pytest

from gpu_cases import dev, host, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grid", [(9, 7, 8), (4, 5, 6), (18, 14, 10), (34, 10, 10), (48, 40, 32),
                                  (144, 16, 16), (256, 16, 24)],
                         ids=lambda g: "x".join(map(str, g)))
@pytest.mark.parametrize("Re", [5.0, 500.0])
def test_predictor_matches_oracle(cuda_device, grid, Re):
    from oracle import mac, step
    from paper_2501_15314_gb300.api import IBMSolver
    nx, ny, nz = grid
    h, dt = 1.0 / nx, 0.004
    g = mac.Grid(nx, ny, nz, h)
    rng = np.random.default_rng(nx + 5 * ny + int(Re))
    mask = g.interior_face_mask_packed()
    u_n, u_nm1, f = (rng.standard_normal(g.n_faces) * mask for _ in range(3))
    p_n = rng.standard_normal(g.m)
    ref = step.step(g, Re, dt, np.zeros((3, 0)), np.zeros(0), f, u_n=u_n, u_nm1=u_nm1, p_n=p_n,
                    rtol=1e-13)
    s = IBMSolver(nx, ny, nz, h, Re=Re, dt=dt)
    none = dev(np.zeros(1))
    out, st = s.step(dev(u_n), dev(u_nm1), dev(p_n), none, none, dev(f), precond_prec=0,
                     rtol=1e-13, helm_rtol=1e-14, helm_maxit=12)
    assert st["helm_relres"] <= 1e-14
    for k in ("u", "p"):
        assert rel(host(out[k]), ref[k]) < 1e-10, (k, rel(host(out[k]), ref[k]))
    assert np.all(host(out["u"])[~mask] == 0.0)
    s.close()
