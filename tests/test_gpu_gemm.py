"""The contraction kernels (csrc/gemm.cu) through an inner product of two-core
trains, whose first step is the r x s product of the first cores over their
mode of n values: sizes next to the tiles' edges (4, 8, 16, 64 rows or columns, 16,
32, 64 of k), thin and tall ones, and those with K split over CTAs.

Tolerance: sums of n, r and s products in some order have an error of about
sqrt(n + r + s) u times the product of the cores' norms; 20 times that."""
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


SHAPES = [(1, 1, 1), (3, 4, 5), (4, 4, 63), (5, 3, 64), (4, 17, 65), (8, 8, 16), (9, 7, 33), (16, 16, 15), (17, 33, 31),
          (64, 4, 2), (65, 5, 3), (4, 65, 2), (70000, 3, 2), (2, 70000, 3), (300, 2, 9), (150, 150, 40), (200, 130, 17),
          (3, 3, 700), (33, 31, 1000), (12, 100, 260), (640, 512, 24)]


@pytest.mark.parametrize("r,s,n", SHAPES)
@pytest.mark.parametrize("fp32", [False, True])
def test_dot_of_two_core_trains(Q, ctx, r, s, n, fp32):
    rng = np.random.default_rng(r * 7 + s * 3 + n)
    kind = np.complex64 if fp32 else np.complex128
    rand = lambda *sh: (rng.standard_normal(sh) + 1j * rng.standard_normal(sh)).astype(kind)
    x, y = [rand(1, n, r), rand(r, 2, 1)], [rand(1, n, s), rand(s, 2, 1)]
    dt = Q.C64 if fp32 else Q.C128
    v = Q.tt_dot(ctx, Q.TT.from_cores(ctx, x, dt), Q.TT.from_cores(ctx, y, dt))
    full = [a[0].astype(np.complex128) @ b[:, :, 0].astype(np.complex128) for a, b in (x, y)]
    scale = math.prod(float(np.linalg.norm(c.astype(np.complex128))) for c in x + y)
    u = 2.0 ** -24 if fp32 else 2.0 ** -53
    assert abs(v - np.vdot(full[0], full[1])) <= 20 * math.sqrt(r + s + n) * u * scale


@pytest.mark.parametrize("K", [8, 40, 256, 1000, 4096])
@pytest.mark.parametrize("value", [0.7, 1.1])
def test_long_sums_of_one_sign(Q, ctx, K, value):
    """A sum of K equal values, whose roundings all go the same way: runs of 8 and the sum of the runs
    round by at most (8 + K / 8) u; one chain is off by 41, 167, 680 u at K = 256, 1000, 4096."""
    import torch
    M, N = 70, 66
    a = torch.full((M, K), value, dtype=torch.complex64, device="cuda")
    b = torch.ones(K, N, dtype=torch.complex64, device="cuda")
    c = torch.empty(M, N, dtype=torch.complex64, device="cuda")
    Q.qtt_cgemm(ctx, M, N, K, a.data_ptr(), b.data_ptr(), c.data_ptr(), engine=0)
    ref = K * float(np.float32(value))
    assert float((c.to(torch.complex128) - ref).abs().max()) <= (8 + K / 8) * 2.0 ** -24 * ref
