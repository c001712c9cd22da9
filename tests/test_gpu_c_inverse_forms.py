"""C^{-1} = (R^T R)^{-1} where its conjugate gradients take one form or the
other: the last marker count of the rows form and the first of the spread form
(a lane group holds at most four rows; 8192 and 8193, which other tests have,
are no limit of it), the last of the one-launch forms and the first solved kernel
by kernel, counts that fill the third and fourth rows, cells with more than the
32 entries a warp reads at once, the two sets too dense for rows (by the cells'
entries, and by the rows' own length), and rows formed again when the markers
change.

C s is recomputed with the library's own spread and interpolation.  Bounds: at
marker spacing h as for the sizes below the limit, 2.2e-16 ||s|| sqrt(500)
with ||s|| < 22 / 1.8e-3 ||t||, 3e-12 over the 1e-13 asked for.  The dense sets'
C is singular; t = C y, so that the solve has a solution, is asked to 1e-6, and
the recursive residual departs from the true one by at most 2.2e-16 ||C|| ||s||
a step, ||C|| < 600 / 8 (the entries of a row), ||s|| < 8 ||t|| for a random y
(C's diagonal is 1/8), over 20000 steps: 3e-9."""
import numpy as np
import pytest

from gpu_cases import dev, host
from paper_2501_15314_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def _limit():
    """Largest marker count of the rows form: 16 warps of 8 rows, 4 times, per SM."""
    import torch
    return torch.cuda.get_device_properties(0).multi_processor_count * 16 * 8 * 4 // 3


@pytest.mark.parametrize("which", ["rounds3", "rounds4", "last_rows", "first_spread",
                                   "last_one_launch", "first_launched"])
def test_large_counts(cuda_device, which):
    from paper_2501_15314_gb300.api import IBMSolver
    count = {"rounds3": _limit() * 5 // 8, "rounds4": _limit() * 7 // 8, "last_rows": _limit(),
             "first_spread": _limit() + 1, "last_one_launch": 150000, "first_launched": 150001}[which]
    n = 128 if count < 100000 else 256
    s = IBMSolver(n)
    s.set_markers(dev(wl.fibonacci_sphere(count, float(np.sqrt(count / (4.0 * np.pi))) / n,
                                          [0.5, 0.48, 0.51])))
    t = dev(np.random.default_rng(count).standard_normal(3 * count))
    x, it = s.apply_c_inverse(t, c_rtol=1e-13, c_maxit=2000)
    r = t - s.interp(s.spread(x))
    assert float(r.norm() / t.norm()) < 3e-12
    if which == "first_launched":   # its own end tests, host-side
        from paper_2501_15314_gb300 import _lib
        with pytest.raises(_lib.IBMError) as e:
            s.apply_c_inverse(t, c_rtol=1e-13, c_maxit=6)
        assert e.value.status == _lib.IBM_ERR_NOT_CONVERGED
        x, it = s.apply_c_inverse(0.0 * t)
        assert it == 0 and float(x.abs().max()) == 0.0
        t[5] = np.nan
        with pytest.raises(_lib.IBMError) as e:
            s.apply_c_inverse(t)
        assert e.value.status == _lib.IBM_ERR_NAN
    s.close()


def _dense(which, n=32):
    """Markers on an n^3 grid."""
    rng = np.random.default_rng(8)
    h = 1.0 / n
    cell = np.array([[0.5], [0.47], [0.44]])
    if which == "cell_of_100":       # rows form; 100 entries in the shared cells
        return np.concatenate([cell + rng.uniform(0.0, 0.9 * h, (3, 100)),
                               wl.fibonacci_sphere(700, 0.25, [0.5, 0.5, 0.5])], axis=1)
    if which == "entries":           # 600 entries a cell
        return cell + rng.uniform(0.0, 0.9 * h, (3, 600))
    if which == "rows_of_two":       # 90 in a row, too long for two rows a lane group
        return 10 * h + rng.uniform(0.0, 28 * h, (3, 7000))
    # "rows": one and a half markers a cell, about 360 in a row
    return 8 * h + rng.uniform(0.0, 16 * h, (3, 6144))


@pytest.mark.parametrize("which,n", [("cell_of_100", 32), ("entries", 32), ("rows", 32),
                                     ("rows_of_two", 64)])
def test_dense_markers(cuda_device, which, n):
    from paper_2501_15314_gb300.api import IBMSolver
    X = _dense(which, n)
    s = IBMSolver(n)
    s.set_markers(dev(X))
    y = dev(np.random.default_rng(9).standard_normal(X.size))
    t = s.interp(s.spread(y))
    assert float(y.norm() / t.norm()) < 8.0
    for _ in range(2):   # the second with what the first formed
        x, it = s.apply_c_inverse(t, c_rtol=1e-6, c_maxit=20000)
        assert it > 0
        r = t - s.interp(s.spread(x))
        assert float(r.norm() / t.norm()) < 1e-6 + 3e-9
    s.close()


def test_rows_follow_the_markers(cuda_device):
    """One solver through sets of the same, a smaller, a larger and again the
    first count, a dense one between, against a fresh solver each: same bits."""
    from paper_2501_15314_gb300.api import IBMSolver
    ball = lambda n, c: wl.fibonacci_sphere(n, 0.22, c)   # noqa: E731
    sets = [ball(500, [0.5, 0.5, 0.5]), ball(500, [0.46, 0.5, 0.53]), ball(120, [0.5, 0.4, 0.5]),
            _dense("entries"), ball(800, [0.5, 0.5, 0.5]), ball(500, [0.5, 0.5, 0.5])]
    s = IBMSolver(32)
    for k, X in enumerate(sets):
        s.set_markers(dev(X))
        r = IBMSolver(32)
        r.set_markers(dev(X))
        t = s.interp(s.spread(dev(np.random.default_rng(k).standard_normal(X.size))))
        x, it = s.apply_c_inverse(t, c_rtol=1e-6, c_maxit=2000)
        y, it2 = r.apply_c_inverse(t, c_rtol=1e-6, c_maxit=2000)
        assert it == it2
        np.testing.assert_array_equal(host(x), host(y))
        r.close()
    s.close()
