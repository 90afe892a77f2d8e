"""The cluster QR kernel (csrc/qr.cu) at the edges of its tiles: row counts next
to a 32-row slice and to the instances' limits, column counts next to a panel,
to the one-CTA limit and to a second panel per CTA, wide and tall shapes, and
matrices whose squares leave the range of their type.

Tolerances: a Householder QR of a k-column matrix has a backward error of a
few k u ||A|| at worst and about sqrt(k) u ||A|| in practice; 20 sqrt(k) u
(u = 2^-24 or 2^-53, k <= 512) bounds both quantities compared here."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def Q():
    from paper_2512_07811_gb300 import qtt
    return qtt


@pytest.fixture(scope="module")
def ctx(Q):
    return Q.Context(0)


def _rand(rng, *shape):
    return rng.standard_normal(shape) + 1j * rng.standard_normal(shape)


def _tol(k, fp32):
    return 20 * math.sqrt(k) * (2.0 ** -24 if fp32 else 2.0 ** -53)


SHAPES = [(1, 1), (5, 3), (16, 16), (31, 17), (32, 33), (33, 8), (65, 9), (97, 128), (129, 130), (160, 24), (193, 192),
          (257, 136), (288, 129), (289, 40), (384, 257), (385, 65), (512, 260), (40, 300)]


@pytest.mark.parametrize("m,n", SHAPES)
@pytest.mark.parametrize("fp32", [False, True])
def test_norm_of_a_two_core_train(Q, ctx, m, n, fp32):
    """||A b|| by the R factor of A (m x n): the norm of the train (A, b)."""
    rng = np.random.default_rng(m * 1000 + n)
    A, b = _rand(rng, 1, m, n), _rand(rng, n, 3, 1)
    dt = Q.C64 if fp32 else Q.C128
    cast = (lambda a: a.astype(np.complex64)) if fp32 else (lambda a: a)
    A, b = cast(A), cast(b)
    v = Q.tt_norm(ctx, Q.TT.from_cores(ctx, [A, b], dt))
    ref = np.linalg.norm(A[0].astype(np.complex128) @ b[:, :, 0].astype(np.complex128))
    # the error relative to ||A|| ||b||, which random factors exceed ||A b|| by at most sqrt(min(m, n))
    scale = np.linalg.norm(A) * np.linalg.norm(b) / math.sqrt(n)
    assert abs(v - ref) <= _tol(max(m, n), fp32) * max(ref, scale)


# (the identity operator of the second site batches m n contractions: at most 65535)
@pytest.mark.parametrize("m,n", [s for s in SHAPES if s[0] * s[1] <= 65535] + [(512, 120), (300, 200)])
@pytest.mark.parametrize("fp32", [False, True])
def test_projection_onto_an_explicit_q(Q, ctx, m, n, fp32):
    """Sketched rounding with the exact right basis: Q Q^H (A B) = A B for the
    explicit Q of the m x n sketched unfolding."""
    rng = np.random.default_rng(m * 1000 + n + 7)
    r = min(5, n)
    dt = Q.C64 if fp32 else Q.C128
    x = [_rand(rng, 1, m, r), _rand(rng, r, n, 1)]
    sk = [_rand(rng, 1, m, n), np.eye(n).reshape(n, n, 1).astype(np.complex128)]
    y, _ = Q.tt_round_sketched(ctx, [(1.0, None, Q.TT.from_cores(ctx, x, dt))], Q.TT.from_cores(ctx, sk, dt), 0.0)
    a, b = [c.astype(np.complex128) for c in y.cores()]
    full, ref = a[0] @ b[:, :, 0], x[0][0] @ x[1][:, :, 0]
    # FP32: the cores are rounded to single precision first, and the SVD sweep adds its own few units
    assert np.linalg.norm(full - ref) <= 4 * _tol(max(m, n), fp32) * np.linalg.norm(ref)


# FP32 matrices too wide for a cluster's shared memory: the blocked kernel's instances, then the panel kernel
WIDE = [(120, 3000), (250, 1500), (288, 1300), (400, 700), (500, 700)]


@pytest.mark.parametrize("m,n", WIDE)
def test_norm_of_a_wide_train(Q, ctx, m, n):
    test_norm_of_a_two_core_train(Q, ctx, m, n, True)


@pytest.mark.parametrize("m,n", WIDE)
def test_projection_of_a_wide_sketch(Q, ctx, m, n):
    """The explicit Q (m x m) of an m x n sketched unfolding of rank 2: Q Q^H = 1."""
    rng = np.random.default_rng(m * 1000 + n + 9)
    x = [_rand(rng, 1, m, 2), _rand(rng, 2, 2, 1)]
    sk = [_rand(rng, 1, m, n), _rand(rng, n, 2, 1)]
    y, _ = Q.tt_round_sketched(ctx, [(1.0, None, Q.TT.from_cores(ctx, x, Q.C64))], Q.TT.from_cores(ctx, sk, Q.C64), 0.0)
    a, b = [c.astype(np.complex128) for c in y.cores()]
    full, ref = a[0] @ b[:, :, 0], x[0][0] @ x[1][:, :, 0]
    assert np.linalg.norm(full - ref) <= 4 * _tol(m, True) * np.linalg.norm(ref)


@pytest.mark.parametrize("scale", [1e-28, 1e-15, 1e15])
def test_fp32_range(Q, ctx, scale):
    """Squares of the entries leave the FP32 range; the kernel scales by a power of two."""
    rng = np.random.default_rng(3)
    A, b = _rand(rng, 1, 70, 20) * scale, _rand(rng, 20, 3, 1) / scale
    v = Q.tt_norm(ctx, Q.TT.from_cores(ctx, [A, b], Q.C64))
    ref = np.linalg.norm(A[0] @ b[:, :, 0])
    assert abs(v - ref) <= _tol(70, True) * np.linalg.norm(A) * np.linalg.norm(b)
