"""Error of complex64 solves against 64-bit ones, over geometries and sketch
seeds: what the single-precision arithmetic of a solve and of its operators
adds up to.

Bounds.  Solves: with arithmetic in 64 bits and every train stored in complex64,
C_eff of these problems is off by 0.4e-6 rms.  Contractions with runs of 8 terms
and factorisations that leave the vectors' norms to storage add about three times
that (their error and storage's are of the same size, over three kinds of kernel),
and a bound of 2e-6 leaves room for the scatter of 24 solves.  Operators: a
Green operator of 13 sites stored in complex64 is off by 2e-7 (2-norm), by
about 5e-7 with the errors of its factorisations and products; the fixed
point carries that on by less than 1 / (1 - 0.82) (contrast 10), over four
iterations 2.5 times at most, half of it at the mean: 1e-6 of the strain, rms."""
import math

import numpy as np
import pytest

from paper_2512_07811_gb300 import inputs as I

pytestmark = pytest.mark.gpu

N = 16


@pytest.fixture(scope="module")
def Q():
    from paper_2512_07811_gb300 import qtt
    return qtt


@pytest.fixture(scope="module")
def ctx(Q):
    return Q.Context(0)


def _voigt(lam, mu):
    C = np.zeros((6, 6))
    C[:3, :3] = lam
    C[range(3), range(3)] += 2 * mu
    C[range(3, 6), range(3, 6)] = mu
    return C


def _problem(Q, seed):
    rng = np.random.default_rng(seed)
    rows = I.sphere_rows(float(rng.uniform(0.17, 0.23)), tuple(rng.uniform(0.3, 0.7, 3)))
    l1, m1 = I.lame_from_young(1.0, 0.3)
    l2, m2 = I.lame_from_young(float(rng.uniform(8.0, 12.0)), 0.3)
    return Q.Ellipsoids(rows, (N, N, N)), (l1, m1, l2, m2), _voigt(0.5 * (l1 + l2), 0.5 * (m1 + m2))


def _solve(Q, ctx, problem, op_prec, prec, seed, **kw):
    geo, moduli, C0 = problem
    ops = Q.ms_setup(ctx, geo, "elastic", moduli, C0, op_tol=1e-6, op_prec=op_prec)
    return Q.ms_homogenize(ctx, geo, "elastic", moduli, C0, tol=0.0, max_rank=128, eps=1e-6, op_tol=1e-6, max_iter=4,
                           min_iter=4, prec=prec, ops=ops, seed=seed, **kw)


def _rms(v):
    return math.sqrt(np.mean(np.square(v)))


def test_operators_in_single_precision(Q, ctx):
    """Strain of the first load case, FP64 solves with operators in either precision."""
    err = []
    for g in range(10):
        e = [Q.contract_voxels(ctx, _solve(Q, ctx, _problem(Q, g), p, Q.PREC_F64, 1, load_mask=1,
                                           return_strain=True)[1].strain, [4] * 3) for p in (Q.PREC_F64, Q.PREC_F32)]
        err.append(np.linalg.norm(e[1] - e[0]) / np.linalg.norm(e[0]))
    assert _rms(err) <= 1e-6


def test_solves_in_single_precision(Q, ctx):
    """C_eff, against the FP64 path with FP64 operators (itself off by 1e-8 at most)."""
    err = []
    for g in range(6):
        problem = _problem(Q, g)
        ref = _solve(Q, ctx, problem, Q.PREC_F64, Q.PREC_F64, 1, lc_workers=6)[0]
        err += [np.linalg.norm(_solve(Q, ctx, problem, Q.PREC_F32, Q.PREC_F32, s, lc_workers=6)[0] - ref) /
                np.linalg.norm(ref) for s in (1, 2, 3, 4)]
    assert _rms(err) <= 2e-6
