"""The SVD step of a rounding (sorted QR, FP64 column rotations started in FP32,
cluster Jacobi; csrc/jacobi.cu) at the edges of its plans: rows next to a
16- or 32-row slice and to the instances' limits, one to many columns per block,
square and tall, and the spectra on which it can go wrong.

A two-core train (U diag(s), W^H) of p modes and rank q has the SVD of its
p x q matrix taken; U, s and W are known.

Tolerances: the backward error of the QR and of the rotations is about
sqrt(k) u ||A|| in practice (k = p + q, u = 2^-24 or 2^-53), as is what rounding
adds to the cosines of the vectors, which the rotations bring below 2 u:
20 sqrt(k) u bounds the entries of the Gram matrix, 40 sqrt(k) u the norm of
the reconstruction's error (two cores) beyond the tail that is cut."""
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


def _unitary(rng, m, n):
    q, r = np.linalg.qr(rng.standard_normal((m, n)) + 1j * rng.standard_normal((m, n)))
    return q * (np.diag(r) / abs(np.diag(r)))


def _spectrum(kind, q, fp32):
    """values, the tolerance to round to, the rank that is left (the others are below a tenth of it in all)"""
    if kind == "graded":  # all kept
        return np.logspace(0, -3 if fp32 else -9, q), 0.0, q
    if kind == "deficient":  # columns of rounding noise, which may be left out
        k = q // 3 + 1
        s = np.zeros(q)
        s[:k] = np.logspace(0, -1 if fp32 else -4, k)
        return s, 1e-4 if fp32 else 1e-8, k
    k = (q + 1) // 2
    s = np.full(q, (1e-6 if fp32 else 1e-12) / math.sqrt(q))
    if kind == "noise":
        s[:k] = np.logspace(0, -1 if fp32 else -4, k)
    elif kind == "equal":  # one value many times: any basis of its space is as good
        s[:k] = 1.0
    else:  # pairs that single precision cannot tell apart
        s[:k] = np.repeat(np.logspace(0, -1, (k + 1) // 2), 2)[:k] * (1 + 1e-9 * (np.arange(k) % 2))
    return s, 1e-4 if fp32 else 1e-8, k


SHAPES = [(1, 1), (2, 2), (5, 3), (16, 16), (17, 15), (32, 32), (33, 31), (64, 33), (65, 64), (96, 48), (97, 97),
          (128, 16), (129, 65), (160, 129), (193, 100), (200, 24), (255, 33), (256, 128), (257, 40), (300, 7)]


@pytest.mark.parametrize("p,q", SHAPES)
@pytest.mark.parametrize("kind", ["graded", "noise", "equal", "pairs", "deficient"])
@pytest.mark.parametrize("fp32", [False, True])
def test_svd_of_a_two_core_train(Q, ctx, p, q, kind, fp32):
    rng = np.random.default_rng(p * 1000 + q)
    s, eps, rank = _spectrum(kind, q, fp32)
    x = [(_unitary(rng, q, q) * s)[None], _unitary(rng, p, q).conj().T[:, :, None]]
    y, info = Q.tt_round(ctx, Q.TT.from_cores(ctx, x, Q.C64 if fp32 else Q.C128), eps)
    assert y.ranks[1] == rank
    a, b = [c.astype(np.complex128) for c in y.cores()]
    b = b[:, :, 0]
    u, tol = (2.0 ** -24 if fp32 else 2.0 ** -53), math.sqrt(p + q)
    assert abs(b @ b.conj().T - np.eye(rank)).max() <= 20 * tol * u
    err = np.linalg.norm(a[0] @ b - x[0][0] @ x[1][:, :, 0])
    assert err <= np.linalg.norm(s[rank:]) + 40 * tol * u * np.linalg.norm(s)


@pytest.mark.parametrize("p,q", [(17, 15), (64, 33), (128, 72)])
@pytest.mark.parametrize("fp32", [False, True])
def test_batch_with_a_rank_per_train(Q, ctx, p, q, fp32):
    """Trains rounded together keep their own ranks; rows beyond them are cropped."""
    rng = np.random.default_rng(p * 1000 + q + 1)
    dt, xs = Q.C64 if fp32 else Q.C128, []
    ranks = [1, q // 2, q]
    for k in ranks:
        s = np.full(q, (1e-6 if fp32 else 1e-12) / math.sqrt(q))
        s[:k] = np.logspace(0, -1, k)
        xs.append([(_unitary(rng, q, q) * s)[None], _unitary(rng, p, q).conj().T[:, :, None]])
    ys, _ = Q.tt_round_batch(ctx, [Q.TT.from_cores(ctx, x, dt) for x in xs], 1e-4 if fp32 else 1e-8)
    u, tol = (2.0 ** -24 if fp32 else 2.0 ** -53), math.sqrt(p + q)
    for k, x, y in zip(ranks, xs, ys):
        assert y.ranks[1] == k
        a, b = [c.astype(np.complex128) for c in y.cores()]
        ref = x[0][0] @ x[1][:, :, 0]
        assert np.linalg.norm(a[0] @ b[:, :, 0] - ref) <= (1e-6 if fp32 else 1e-12) + 40 * tol * u * np.linalg.norm(ref)


@pytest.mark.parametrize("m,n", [(23, 40), (30, 24), (64, 64), (100, 130), (130, 70)])
@pytest.mark.parametrize("kind", ["graded", "noise", "deficient"])
def test_svd_of_a_dense_matrix(Q, ctx, m, n, kind):
    """TT-SVD of an m x n array: left vectors and the values they are cut by."""
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(m * 1000 + n + 2)
    q = min(m, n)
    s, eps, rank = _spectrum(kind, q, False)
    A = _unitary(rng, m, q) * s @ _unitary(rng, n, q).conj().T
    d = torch.tensor(A, device="cuda")
    y = Q.tt_from_dense(ctx, d.data_ptr(), [m, n], eps)
    assert y.ranks[1] == rank
    a, b = y.cores()
    tol = math.sqrt(m + n) * 2.0 ** -53
    assert abs(a[0].conj().T @ a[0] - np.eye(rank)).max() <= 20 * tol
    assert np.linalg.norm(a[0] @ b[:, :, 0] - A) <= np.linalg.norm(s[rank:]) + 40 * tol * np.linalg.norm(s)


def test_zero_tolerance(Q, ctx):
    """No noise is left out at a zero tolerance."""
    rng = np.random.default_rng(5)
    s = np.zeros(60)
    s[:20] = np.logspace(0, -3, 20)
    x = [(_unitary(rng, 60, 60) * s)[None], _unitary(rng, 80, 60).conj().T[:, :, None]]
    y, info = Q.tt_round(ctx, Q.TT.from_cores(ctx, x, Q.C128), 0.0)
    assert y.ranks[1] >= 20 and info.tail == 0.0


@pytest.mark.parametrize("sketched", [False, True])
def test_norms_of_rounded_cores_fp32(Q, ctx, sketched):
    """Cores 2..d of a complex64 rounding have rows of norm 1 to what storing their entries allows.  What storing
    leaves is taken from the rows themselves (normalised in FP64, rounded); forming the sum of squares adds the
    rounding of each square, 0.5 u rms where one entry makes up the row, independent of it."""
    rng = np.random.default_rng(5)
    r = [1] + [min(40, 2 ** k, 2 ** (14 - k)) for k in range(1, 14)] + [1]
    x = [rng.standard_normal((r[k], 2, r[k + 1])) + 1j * rng.standard_normal((r[k], 2, r[k + 1])) for k in range(14)]
    x = Q.TT.from_cores(ctx, [(c / np.linalg.norm(c)).astype(np.complex64) for c in x], Q.C64)
    if sketched:
        w = [1] + [min(48, 2 ** k, 2 ** (14 - k)) for k in range(1, 14)] + [1]
        S = Q.TT.from_cores(ctx, [rng.standard_normal((w[k], 2, w[k + 1])).astype(np.complex64) for k in range(14)],
                            Q.C64)
        y, _ = Q.tt_round_sketched(ctx, [(1.0, None, x)], S, 1e-6)
    else:
        y, _ = Q.tt_round(ctx, x, 1e-6)
    norm2 = lambda m: (abs(m.astype(np.complex128)) ** 2).sum(1) - 1  # noqa: E731
    off, stored = [], []
    for c in y.cores()[1:]:
        m = c.astype(np.complex128).reshape(c.shape[0], -1)
        off.append(norm2(m))
        stored.append(norm2((m / np.linalg.norm(m, axis=1, keepdims=True)).astype(np.complex64)))
    rms = lambda v: math.sqrt((np.concatenate(v) ** 2).mean())  # noqa: E731
    assert rms(off) <= math.hypot(rms(stored), 0.5 * 2.0 ** -24)


def test_cosines_left_by_the_last_sweep(Q, ctx):
    """Two columns whose cosine is 6e-9: small enough for the quadratic regime, large enough that a rotation
    from a 20-bit angle alone would leave up to 3e-15.  Rotations stop below 2 u (a threshold by exponents); the
    two stored vectors' entries, each good to 2 u (scaled, rounded), add 4 u at most: 6 u."""
    rng = np.random.default_rng(11)
    worst = 0.0
    for ratio in np.linspace(0.2, 0.6, 60):
        # the first column is the largest and parallel to e_1, so that the QR leaves the rows as they are
        c = _unitary(rng, 7, 2).conj().T * np.array([[0.3], [1.0]])
        c[1] += 6e-9 / 0.3 * c[0] / 0.3
        c = np.concatenate([[[0.95], [0.0]], c], axis=1)
        c = c / np.linalg.norm(c, axis=1, keepdims=True) * np.array([[1.0], [ratio]])
        y, _ = Q.tt_round(ctx, Q.TT.from_cores(ctx, [np.eye(2)[None], c[:, :, None]], Q.C128), 0.0)
        b = y.cores()[1][:, :, 0].astype(np.clongdouble)
        assert b.shape == (2, 8)
        worst = max(worst, float(abs((b[0].conj() * b[1]).sum())))
    assert worst <= 6 * 2.0 ** -53


def test_profile_counts_the_fp32_start(Q, ctx):
    """An FP64 SVD of 64 columns starts with FP32 rotations: a Jacobi launch of its own in the profiler."""
    rng = np.random.default_rng(2)
    x = Q.TT.from_cores(ctx, [(_unitary(rng, 64, 64) * np.logspace(0, -6, 64))[None],
                              _unitary(rng, 64, 64).conj().T[:, :, None]], Q.C128)
    ctx.profile(True)
    try:
        Q.tt_round(ctx, x, 1e-9)
        rows = {r["variant"]: r for r in ctx.profile_shapes("jacobi")}
        total = ctx.profile_read("jacobi")
    finally:
        ctx.profile(False)
    assert sorted(rows) == [0, 1] and total["launches"] == 2
    for r in rows.values():
        assert r["dims"] == (64, 64, 0) and r["launches"] == 1 and r["ms"] > 0 and r["flops"] > 0
    # the sweeps of the two: several in FP32, then two or three
    assert rows[1]["flops"] > rows[0]["flops"]
