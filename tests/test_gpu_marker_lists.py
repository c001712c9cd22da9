"""The marker lists from one build to the next: one marker, cells with more
entries than the register sort takes (64), several blocks of cells, sets that
shrink, grow and move, and a refused set between two accepted ones.  R, R^T and
S~ against the oracle's matrices at 1e-13 (the repository's bound for
operators), and bit for bit the same after other sets have come between."""
import numpy as np
import pytest

from gpu_cases import dev, host, rel
from paper_2501_15314_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

N = (48, 40, 32)
H = 1.0 / 48


def _sets():
    rng = np.random.default_rng(3)
    one = np.array([[0.31], [0.4], [0.29]])
    # 150 markers within one cell: segments of 150 entries
    dense = np.array([[0.5], [0.4], [0.3]]) + rng.uniform(0.0, 0.9 * H, (3, 150))
    # a taps' distance of exactly half a cell, and markers on faces and centres
    exact = H * np.array([[10.0, 10.5, 11.0, 12.5], [9.5, 9.0, 9.5, 14.0], [8.0, 8.5, 8.5, 9.0]])
    ball = wl.fibonacci_sphere(700, 0.2, [0.5, 0.42, 0.33])
    line = np.stack([rng.uniform(0.06, 0.94, 400), rng.uniform(0.06, 0.76, 400),
                     rng.uniform(0.06, 0.6, 400)])
    return [one, dense, exact, ball, line, one, ball]


def _check(s, g, X, rng):
    from oracle import delta, mac
    R = delta.regularization_matrix(g, X)
    F, u = rng.standard_normal(X.size), rng.standard_normal(g.n_faces)
    u *= g.interior_face_mask_packed()
    v = rng.standard_normal(g.m)
    B = R.T @ mac.apply_G(g, v)
    S = mac.apply_GT(g, mac.apply_G(g, v)) + 2.0 * mac.apply_GT(g, R @ B)
    out = [host(s.interp(dev(u))), host(s.spread(dev(F))), host(s.apply_schur(dev(v)))]
    assert rel(out[0], R.T @ u) < 1e-13
    assert rel(out[1], R @ F) < 1e-13
    assert rel(out[2], S) < 1e-13
    return out


def test_marker_lists_over_several_sets(cuda_device):
    from oracle import mac
    from paper_2501_15314_gb300 import _lib
    from paper_2501_15314_gb300.api import IBMSolver
    g = mac.Grid(*N, H)
    s = IBMSolver(*N, H, Re=100.0, dt=0.01)
    first = {}
    for X in _sets():
        s.set_markers(dev(X))
        out = _check(s, g, X, np.random.default_rng(X.shape[1]))
        for a, b in zip(out, first.setdefault(X.shape[1], out)):
            np.testing.assert_array_equal(a, b)
        bad = X.copy()
        bad[1, -1] = 0.01 if X.shape[1] % 2 else np.nan
        with pytest.raises(_lib.IBMError) as e:
            s.set_markers(dev(bad))
        assert e.value.status == _lib.IBM_ERR_MARKER_DOMAIN
    s.close()
