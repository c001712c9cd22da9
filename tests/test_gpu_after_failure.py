"""A solver after a call that failed: nothing of the failed call shows in the
ones that follow, and the marker operators fit the markers that the library
holds then."""
import numpy as np
import pytest

from gpu_cases import dev, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grid", [(12, 8, 8), (16, 8, 8), (20, 12, 8), (18, 14, 10), (9, 7, 8)],
                         ids=lambda g: "x".join(map(str, g)))
def test_step_after_an_overflowing_one(cuda_device, grid):
    """The right-hand side 4 u^n / (2 dt) = 4e31 is finite in FP64 and past the
    range of its FP32 parts (2^101), so the predictor ends with IBM_ERR_NAN;
    a valid step after it gives the bits of one on a fresh solver."""
    from paper_2501_15314_gb300 import _lib
    from paper_2501_15314_gb300.api import IBMSolver
    nx, ny, nz = grid
    rng = np.random.default_rng(nx)
    none = dev(np.zeros(1))

    def solver():
        return IBMSolver(nx, ny, nz, 1.0 / nx, Re=50.0, dt=5e-4)

    def step(s, u, **kw):
        return s.step(u, zero, cells, none, none, f, raise_on_error=False, with_advection=0, **kw)

    a, b = solver(), solver()
    zero, cells = dev(np.zeros(a.nf)), dev(np.zeros(a.m))
    f = dev(rng.standard_normal(a.nf))
    good = dev(rng.standard_normal(a.nf))
    ref, st = step(a, good)
    assert st["status"] == _lib.IBM_OK
    for _ in range(2):
        _, st = step(b, dev(np.full(a.nf, 1e28)))
        assert st["status"] == _lib.IBM_ERR_NAN
        out, st = step(b, good)
        assert st["status"] == _lib.IBM_OK
        for k in ("u", "p"):
            np.testing.assert_array_equal(host(out[k]), host(ref[k]))
    a.close()
    b.close()


N = 24


def _ball(count, centre, radius=0.15):
    from paper_2501_15314_gb300 import workloads as wl
    return wl.fibonacci_sphere(count, radius, centre)


def _two_way(s, count, centre, body=0, **kw):
    import torch
    from paper_2501_15314_gb300.api import RigidSpheres
    sp = RigidSpheres([0.15], [1.1], [centre])
    u, p = dev(np.zeros(s.nf)), dev(np.zeros(s.m))
    f = dev(np.random.default_rng(1).standard_normal(s.nf))
    return s.fsi_step(sp, dev(_ball(count, [0.0, 0.0, 0.0])),
                      dev(np.full(count, body)).to(torch.int32), u, u, p,
                      dev(np.zeros(3 * count)), f, tol=1e-30, max_inner=1, **kw)


def _used(n):
    """Leaves a block of n FP64 values that are not zero with the allocator."""
    import torch
    for _ in range(4):
        t = torch.full((n,), 7.0, dtype=torch.float64, device="cuda")
    del t


def _solver():
    from paper_2501_15314_gb300.api import IBMSolver
    return IBMSolver(N, Re=50.0, dt=2e-3)


def test_marker_operators_after_a_refused_two_way_step(cuda_device):
    """The body's markers reach a wall: the library holds none, and the
    operators return zeros."""
    from paper_2501_15314_gb300 import _lib
    s = _solver()
    u = dev(np.random.default_rng(2).standard_normal(s.nf))
    p = dev(np.random.default_rng(3).standard_normal(s.m))
    s.set_markers(dev(_ball(90, [0.5, 0.5, 0.5])))
    out, st = _two_way(s, 150, [0.12, 0.5, 0.5], raise_on_error=False)
    assert st["status"] == _lib.IBM_ERR_MARKER_DOMAIN
    assert s.n_markers == 150   # the count asked for
    _used(3 * s.n_markers)
    assert float(s.interp(u).abs().max()) == 0.0
    _used(3 * s.n_markers)
    assert float(s.force_correction(p, dev(np.ones(3 * s.n_markers))).abs().max()) == 0.0
    s.close()


def test_marker_operators_after_a_two_way_step_with_a_bad_body(cuda_device):
    """Refused before the markers move: those set before it stay."""
    from paper_2501_15314_gb300 import _lib
    s = _solver()
    u = dev(np.random.default_rng(2).standard_normal(s.nf))
    s.set_markers(dev(_ball(90, [0.5, 0.5, 0.5])))
    ref = host(s.interp(u))
    out, st = _two_way(s, 150, [0.5, 0.5, 0.5], body=3, raise_on_error=False)
    assert st["status"] == _lib.IBM_ERR_ARG
    np.testing.assert_array_equal(host(s.interp(u)), ref)
    s.close()


@pytest.mark.parametrize("count", [150, 60])
def test_marker_operators_after_an_unfinished_two_way_step(cuda_device, count):
    """IBM_ERR_NOT_CONVERGED, raised: the step's markers are the library's."""
    from paper_2501_15314_gb300 import _lib
    s = _solver()
    u = dev(np.random.default_rng(2).standard_normal(s.nf))
    s.set_markers(dev(_ball(90, [0.5, 0.5, 0.5])))
    with pytest.raises(_lib.IBMError) as e:
        _two_way(s, count, [0.5, 0.45, 0.5])
    assert e.value.status == _lib.IBM_ERR_NOT_CONVERGED
    assert s.n_markers == count   # before any operator writes that many
    U = host(s.interp(u))
    r = _solver()
    r.set_markers(dev(_ball(count, [0.5, 0.45, 0.5])))
    np.testing.assert_array_equal(U, host(r.interp(u)))
    r.close()
    s.close()
