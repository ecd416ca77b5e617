"""The wall density of a one-column channel of a batch (Eq. 9) is summed across velocity rows and
normalised in FP64, as in the other batch kernels: one step without collisions, in which the
populations that come from a wall are a chain of FP32 operations around that one number, bit for bit."""
import math
from fractions import Fraction

import numpy as np
import pytest

from oracle.march import COUETTE, make_problem as oracle_problem
from paper_1308_0692_gb300 import lbm
from paper_1308_0692_gb300.inputs import random_state

f32 = np.float32


def _fma(a, b, c):
    """FP32 fma of float32 scalars: the exact value, rounded once (subnormals do not occur)."""
    v = Fraction(float(a)) * Fraction(float(b)) + Fraction(float(c))
    if v == 0:
        return f32(0)
    e = math.frexp(abs(float(v)))[1] - 24            # the value lies in [2^(e + 23), 2^(e + 24))
    q = v / Fraction(2) ** e
    n, r = divmod(q.numerator, q.denominator)
    twice = 2 * r
    n += twice > q.denominator or (twice == q.denominator and n % 2)
    return f32(math.ldexp(n, e))


def from_walls(p, xi, w, h, fp64=True):
    """[2][M/2][M]: the values one step gives the bottom cell's up-moving rows and the top cell's
    down-moving rows.  fp64 False: the density by products, sums and factor in FP32 pairs."""
    m, half = len(xi), len(xi) // 2
    inv = 1.0 / float(np.sum(xi[half:] * w[half:]))
    cy = f32(p.coeffs["dt"] / p.coeffs["dy"])
    h = h.astype(f32).reshape(m, m, p.ny)
    out = np.empty((2, half, m), dtype=f32)
    for side, (cell, leaving, entering) in enumerate(((0, range(half), range(half, m)), (p.ny - 1, range(half, m), range(half)))):
        dens, pair = 0.0, 0.0
        for iy in leaving:
            s = f32(0)
            for ix in range(m):
                s = f32(s + h[iy, ix, cell])
            dens += abs(xi[iy]) * float(s)
            pair += float(abs(f32(xi[iy]))) * float(s)
        rho = f32(dens * inv) if fp64 else f32(pair * float(f32(inv)))
        for r, iy in enumerate(entering):
            for ix in range(m):
                ghost = f32(f32(f32(w[ix]) * f32(w[iy])) * rho)
                old = h[iy, ix, cell]
                out[side, r, ix] = _fma(f32(abs(f32(xi[iy])) * cy), f32(ghost - old), old)
    return out


def _channels(n_half):
    probs = [oracle_problem("half", n_half, COUETTE, 1, ny, math.inf, 0.0, 0.0) for ny in range(2, 34)]
    return [(p, random_state(p.n, p.ncells, seed=900 + p.ny).astype(f32).astype(np.float64)) for p in probs]


def _rule(p):
    m = int(round(math.sqrt(p.n)))
    return p.xi_x[:m], p.w.reshape(m, m).sum(axis=0), m          # velocity iy M + ix; the weights sum to one


@pytest.mark.parametrize("n_half", [2, 4])
def test_the_channels_tell_the_two_densities_apart(n_half):
    differ = 0
    for p, h in _channels(n_half):
        xi, w, _ = _rule(p)
        differ += not np.array_equal(from_walls(p, xi, w, h), from_walls(p, xi, w, h, fp64=False))
    assert differ >= 4


@pytest.mark.gpu
@pytest.mark.parametrize("n_half", [2, 4])
def test_wall_density_in_fp64(n_half):
    torch = pytest.importorskip("torch")
    vs = lbm.lbm_make_velocity_set(lbm.LBM_HALF_RANGE_GH, n_half)
    cases = _channels(n_half)
    b = lbm.lbm_batch_init(vs, [lbm.make_problem(COUETTE, 1, p.ny, math.inf, 0.0, 0.0, prec=lbm.LBM_FP32_PERTURB,
                                                 residual_every=7) for p, _ in cases], stream=torch.cuda.Stream())
    for i, (_, h) in enumerate(cases):
        lbm.lbm_batch_set_state(b, i, h)
    lbm.lbm_batch_advance(b, 1, 0.0)
    lbm.lbm_batch_poll(b)
    for i, (p, h) in enumerate(cases):
        xi, w, m = _rule(p)
        got = lbm.lbm_batch_get_state(b, i).astype(f32).reshape(m, m, p.ny)
        ref = from_walls(p, xi, w, h)
        assert np.array_equal(got[m // 2:, :, 0], ref[0]) and np.array_equal(got[:m // 2, :, p.ny - 1], ref[1]), p.ny
    b.close()
