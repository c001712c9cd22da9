"""C^{-1} = (R^T R)^{-1} at the sizes where its one-launch conjugate gradients
change form: one marker (one block), fewer markers than threads, both sides of
the marker count above which the directions are written before the spread, and
more marker values than threads in the grid.

C s is recomputed with the library's own spread and interpolation.  Bound: the
recursive residual ends below 1e-13 ||t||, and departs from the true one by a
few roundings of C s per iteration, at most 2.2e-16 ||s|| sqrt(500) <
2.2e-16 x 22 / 1.8e-3 ||t|| = 3e-12 (1.8e-3: the smallest eigenvalue of C at
marker spacing h)."""
import numpy as np
import pytest

from gpu_cases import dev
from paper_2501_15314_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def _solver(n, radius, count):
    from paper_2501_15314_gb300.api import IBMSolver
    s = IBMSolver(n)
    s.set_markers(dev(wl.fibonacci_sphere(count, radius, [0.5, 0.48, 0.51])))
    return s


@pytest.mark.parametrize("n,count", [(16, 1), (16, 170), (48, 1300), (80, 8192), (80, 8193),
                                     (128, 26100)])
def test_c_inverse_residual(cuda_device, n, count):
    # radius: spacing h on the sphere
    radius = float(np.sqrt(count / (4.0 * np.pi))) / n
    s = _solver(n, radius, count)
    t = dev(np.random.default_rng(count).standard_normal(3 * count))
    x, it = s.apply_c_inverse(t, c_rtol=1e-13, c_maxit=2000)
    r = t - s.interp(s.spread(x))
    assert float(r.norm() / t.norm()) < 3e-12
    y, it2 = s.apply_c_inverse(t, c_rtol=1e-13, c_maxit=2000)
    assert it == it2 and bool((x == y).all())   # fixed orders of summation
    s.close()


def test_c_inverse_limits(cuda_device):
    from paper_2501_15314_gb300 import _lib
    s = _solver(16, 0.2, 100)
    t = dev(np.random.default_rng(2).standard_normal(300))
    with pytest.raises(_lib.IBMError) as e:
        s.apply_c_inverse(t, c_rtol=1e-14, c_maxit=3)
    assert e.value.status == _lib.IBM_ERR_NOT_CONVERGED
    x, it = s.apply_c_inverse(dev(np.zeros(300)))
    assert it == 0 and float(x.abs().max()) == 0.0
    bad = np.ones(300)
    bad[7] = np.nan
    with pytest.raises(_lib.IBMError) as e:
        s.apply_c_inverse(dev(bad))
    assert e.value.status == _lib.IBM_ERR_NAN
    s.close()
