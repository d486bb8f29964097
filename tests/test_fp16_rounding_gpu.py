"""Where FP16 storage rounds, bit for bit.  One step of a board is formed again
in numpy from the stored fields with the kernels' FP32 operations (a product
and a fused multiply-add per curl component, one more per update).  Inside the
interior region E takes H~ unrounded; H~ of every node outside it, which the
interior launch forms itself for its halo, must count as its owner stores it.
The plain columns between the x-UPML and the region belong to the slab kernels:
their E takes stored H~ alone (E_y and E_z, which carry no auxiliary there)."""
import numpy as np
import pytest

from paper_1008_2602_gb300 import workloads as W
from test_node_coefficients import library_coefficients
from test_time_blocking_gpu import interior

pytestmark = pytest.mark.gpu

C0, MU0 = 299792458.0, 4.0e-7 * np.pi
F, D = np.float32, np.float64


def _fma(a, b, c):   # the product of two FP32 values is exact in FP64
    return (D(a) * D(b) + D(c)).astype(F)


def _curl(a1, a0, b1, b0, Sa, Sb):   # Sa (a1 - a0) - Sb (b1 - b0)
    return _fma(F(-Sb), b1 - b0, F(Sa) * (a1 - a0))


def _next(v, axis):
    return np.concatenate([v.take(range(1, v.shape[axis]), axis), v.take([-1], axis)], axis)


def _prev(v, axis):
    return np.concatenate([v.take([0], axis), v.take(range(v.shape[axis] - 1), axis)], axis)


def _curl_h(H, S):   # the three components of S curl H~ (axes of a field: z, y, x)
    hx, hy, hz = H
    return [_curl(hz, _prev(hz, 1), hy, _prev(hy, 0), S[1], S[2]), _curl(hx, _prev(hx, 0), hz, _prev(hz, 2), S[2], S[0]),
            _curl(hy, _prev(hy, 2), hx, _prev(hx, 1), S[0], S[1])]


@pytest.mark.parametrize("nx,ny,nz,upml", [(90, 45, 30, 4), (20, 33, 18, 5)])
def test_halo_values_count_as_stored(nx, ny, nz, upml):
    import torch
    assert torch.cuda.is_available()
    from paper_1008_2602_gb300 import solver
    p = W.random_problem(51, nx, ny, nz, upml=upml, n_steps=80)
    s = solver.Solver(p, precision="fp16")
    dt = s.dt
    eps0 = 1.0 / (MU0 * C0 * C0)
    scale = 2.0 ** np.ceil(np.log2(dt * np.abs(p.source_params[:, 0]).max() / eps0))   # the board's storage scale

    def state():   # the stored values, E and H~
        unit = [scale] * 3 + [scale / (MU0 * C0)] * 3
        return [(D(s.field(c)) / unit[c]).astype(np.float16).astype(F) for c in range(6)]

    s.step(70)
    before = state()
    s.step(1)
    after = state()
    s.close()
    S = [F(C0 * dt / d) for d in (p.dx, p.dy, p.dz)]
    ce = library_coefficients(p)[0]
    ex, ey, ez = before[:3]
    curl = [_curl(_next(ez, 1), ez, _next(ey, 0), ey, S[1], S[2]), _curl(_next(ex, 0), ex, _next(ez, 2), ez, S[2], S[0]),
            _curl(_next(ey, 2), ey, _next(ex, 1), ex, S[0], S[1])]
    x0, x1, y0, y1, z0, z1 = interior(p, "fp16")
    I = np.s_[z0:z1, y0:y1, x0:x1]
    mixed = [h.copy() for h in after[3:]]
    for c in range(3):
        exact = before[3 + c] - curl[c]
        assert np.array_equal(exact[I].astype(np.float16), after[3 + c][I].astype(np.float16)), c
        mixed[c][I] = exact[I]
    free = np.ones((3,) + ex.shape, bool)
    for i, j, k, comp in p.sources:
        free[comp, k, j, i] = False
    mix, sto = _curl_h(mixed, S), _curl_h(after[3:], S)
    differ = 0
    for c in range(3):
        E, f = after[c], free[c]
        got = _fma(ce[..., c], mix[c], before[c]).astype(np.float16)
        assert np.array_equal(got[I][f[I]], E[I][f[I]].astype(np.float16)), c
        rounded = _fma(ce[..., c], sto[c], before[c]).astype(np.float16)
        differ += np.count_nonzero(rounded[I] != got[I])
        if c and x0 > upml:
            P = np.s_[z0:z1, y0:y1, upml:x0]
            assert np.array_equal(rounded[P][f[P]], E[P][f[P]].astype(np.float16)), c
    assert differ > 0 and np.any(after[2][I])   # the rounding of H~ shows in E
