"""The FP64 V-cycle, and the FP32 one on grids whose x-extent is no multiple
of four (both run the one-cell level kernels), against the cycle written out
in numpy: Chebyshev smoothing on D^{-1} L with roots on [0.3, 2], 8-cell
averages, trilinear prolongation, pseudo-inverse on the coarsest level.

The grids put the edges of the 32 x 8 tiles and of the marches everywhere: one
warp that ends at a wall, two and five warps per row of which the last is
partial, single-level and two-level grids, and vectors 8 bytes off the 16-byte
boundary.  Bounds: the largest amplification is the coarsest level's inverse,
whose condition number is at most about 4 (17/pi)^2 3 = 350 (17 cells along
its longest axis), so FP64 rounding stays below 350 x 2.2e-16 x 10 = 1e-12 and
FP32 rounding below 350 x 6e-8 = 2e-5."""
import numpy as np
import pytest

from gpu_cases import dev, host, rel

pytestmark = pytest.mark.gpu

GRIDS = [(4, 4, 4), (18, 14, 10), (16, 16, 16), (34, 10, 10), (48, 40, 32), (64, 72, 40),
         (96, 24, 56), (160, 24, 40), (20, 36, 28)]


def lap(x, h):
    out = np.zeros_like(x)
    for ax in range(3):
        g = np.diff(x, axis=ax)
        lo = [slice(None)] * 3
        hi = [slice(None)] * 3
        lo[ax], hi[ax] = slice(0, -1), slice(1, None)
        out[tuple(lo)] -= g
        out[tuple(hi)] += g
    return out / h ** 2


def prolong(x):
    for ax in range(3):
        lo = np.concatenate([x.take([0], ax), x.take(range(x.shape[ax] - 1), ax)], ax)
        hi = np.concatenate([x.take(range(1, x.shape[ax]), ax), x.take([-1], ax)], ax)
        y = np.stack([0.75 * x + 0.25 * lo, 0.75 * x + 0.25 * hi], ax + 1)
        x = y.reshape(x.shape[:ax] + (2 * x.shape[ax],) + x.shape[ax + 1:])
    return x


def vcycle(b, h, pre, post):
    s = b.shape
    if any(k % 2 or k < 4 for k in s) or b.size <= 64:
        A = np.stack([lap(e.reshape(s), h).ravel() for e in np.eye(b.size)])
        return (np.linalg.pinv(A, rcond=1e-10) @ b.ravel()).reshape(s)
    nn = np.zeros(s)
    for ax in range(3):
        lo = [slice(None)] * 3
        hi = [slice(None)] * 3
        lo[ax], hi[ax] = slice(0, -1), slice(1, None)
        nn[tuple(lo)] += 1.0
        nn[tuple(hi)] += 1.0

    def smooth(x, p):
        for i in range(p):
            w = 1.0 / (1.15 + 0.85 * np.cos((2 * i + 1) * np.pi / (2 * p)))
            x = x + w * h ** 2 / nn * (b - lap(x, h))
        return x

    x = smooth(np.zeros(s), pre)
    r = (b - lap(x, h)).reshape(s[0] // 2, 2, s[1] // 2, 2, s[2] // 2, 2).mean((1, 3, 5))
    return smooth(x + prolong(vcycle(r, 2 * h, pre, post)), post)


@pytest.mark.parametrize("grid", GRIDS, ids=lambda g: "x".join(map(str, g)))
@pytest.mark.parametrize("degrees", [(2, 2), (1, 3), (0, 2), (3, 0)], ids=str)
def test_vcycle_matches_numpy(cuda_device, grid, degrees):
    import torch
    from paper_2501_15314_gb300.api import IBMSolver
    nx, ny, nz = grid
    pre, post = degrees
    h = 1.0 / nx
    b = np.random.default_rng(nx + 3 * ny + 7 * nz).standard_normal((nz, ny, nx))
    b -= b.mean()
    ref = vcycle(b, h, pre, post).ravel()
    s = IBMSolver(nx, ny, nz, h, Re=100.0, dt=0.01)
    bd = dev(b.ravel())
    assert rel(host(s.precond(bd, prec=0, pre=pre, post=post)), ref) < 1e-12
    if nx % 4:
        assert rel(host(s.precond(bd, prec=1, pre=pre, post=post)), ref) < 2e-5
    odd = torch.zeros(b.size + 1, dtype=torch.float64, device="cuda")
    out = torch.zeros(b.size + 1, dtype=torch.float64, device="cuda")
    odd[1:] = bd
    s.precond(odd[1:], prec=0, pre=pre, post=post, out=out[1:])
    assert rel(host(out[1:]), ref) < 1e-12
    s.close()
