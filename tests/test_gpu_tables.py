"""Launches that take many cores at once (a table of 48 cores per launch): sums and
sketched sums of trains next to the table's size, and device blocks that a
context keeps for the next call.

Tolerances: an inner product over d cores of rank at most 6 and modes of 2 has
a relative error of about d u times the product of the factors' norms (u = 2^-24
or 2^-53); 20 d u bounds it, also after a rounding sweep of exact rank."""
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


def _train(rng, d, r, fp32):
    rk = [1] + [r] * (d - 1) + [1]
    c = [rng.standard_normal((rk[k], 2, rk[k + 1])) + 1j * rng.standard_normal((rk[k], 2, rk[k + 1])) for k in range(d)]
    c = [a / np.linalg.norm(a) * r ** 0.5 for a in c]
    return [a.astype(np.complex64) for a in c] if fp32 else c


def _dot(x, y):
    e = np.ones((1, 1), dtype=np.complex128)
    for a, b in zip(x, y):
        e = np.einsum("ab,aic,bid->cd", e, a.conj().astype(np.complex128), b.astype(np.complex128), optimize=True)
    return complex(e[0, 0])


@pytest.mark.parametrize("d", [1, 2, 24, 47, 48, 49, 60])
@pytest.mark.parametrize("fp32", [False, True])
def test_sums_of_many_cores(Q, ctx, d, fp32):
    rng = np.random.default_rng(d)
    dt, u = (Q.C64, 2.0 ** -24) if fp32 else (Q.C128, 2.0 ** -53)
    x, y, w = _train(rng, d, 3, fp32), _train(rng, d, 2, fp32), _train(rng, d, 3, fp32)
    a, b = 0.7 - 0.2j, -1.3 + 0.4j
    X, Y, W = [Q.TT.from_cores(ctx, t, dt) for t in (x, y, w)]
    ref = np.conj(a) * _dot(x, w) + np.conj(b) * _dot(y, w)
    scale = (abs(a) * abs(_dot(x, x)) ** 0.5 + abs(b) * abs(_dot(y, y)) ** 0.5) * abs(_dot(w, w)) ** 0.5
    zs = [Q.tt_add(ctx, a, X, b, Y)]
    if d > 1:
        sketch = Q.TT.from_cores(ctx, _train(rng, d, 6, fp32), dt)  # one column beyond the sum's rank
        zs.append(Q.tt_round_sketched(ctx, [(a, None, X), (b, None, Y)], sketch, 0.0)[0])
    for z in zs:
        assert abs(Q.tt_dot(ctx, z, W) - ref) <= 20 * d * u * scale


def test_kept_blocks_are_bounded_and_given_back(Q):
    """Freed blocks are taken again: the device's free memory stays where it was
    after the first rounds, and comes back with the context."""
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(1)
    x = _train(rng, 18, 64, False)
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    ctx = Q.Context(0)
    free = []
    for _ in range(8):
        X = Q.TT.from_cores(ctx, x, Q.C128)
        y, _ = Q.tt_round(ctx, Q.tt_add(ctx, 1.0, X, 1.0, X), 1e-8)
        v = Q.tt_norm(ctx, y)
        del X, y
        torch.cuda.synchronize()
        free.append(torch.cuda.mem_get_info()[0])
    assert abs(v - 2 * abs(_dot(x, x)) ** 0.5) <= 1e-7 * v
    assert min(free[2:]) >= free[1] - (64 << 20)     # nothing accumulates
    assert free0 - free[-1] <= (512 << 20) + (128 << 20)  # the cache's limit and the pool's granularity
    ctx.close()
    torch.cuda.synchronize()
    assert torch.cuda.mem_get_info()[0] >= free0 - (64 << 20)


@pytest.mark.parametrize("d,r,ctrl", [(1, 1, 0), (1, 2, 3), (2, 2, 0), (3, 40, 0), (5, 3, 6), (6, 33, 0), (9, 8, 1), (12, 9, 0),
                                      (14, 32, 0), (11, 40, 6), (4, 600, 0), (13, 1, 0)])
@pytest.mark.parametrize("fp32", [False, True])
def test_read_out_of_a_whole_train(Q, ctx, d, r, ctrl, fp32):
    """Every entry of a train of d bits along one axis: the first and last cores
    are multiplied up on their own, up to bonds of 8 or 32 values."""
    rng = np.random.default_rng(d * 100 + r)
    modes = ([ctrl] if ctrl else []) + [2] * d
    rk = [1] + [r] * (len(modes) - 1) + [1]
    x = [rng.standard_normal((rk[k], n, rk[k + 1])) + 1j * rng.standard_normal((rk[k], n, rk[k + 1]))
         for k, n in enumerate(modes)]
    x = [a / np.linalg.norm(a) * r ** 0.5 for a in x]
    if fp32:
        x = [a.astype(np.complex64) for a in x]
    v = Q.contract_voxels(ctx, Q.TT.from_cores(ctx, x, Q.C64 if fp32 else Q.C128), [d, 0, 0])
    full = np.ones((1, 1), dtype=np.complex128)
    for a in x:
        full = (full @ a.astype(np.complex128).reshape(a.shape[0], -1)).reshape(-1, a.shape[2])
    u = 2.0 ** -24 if fp32 else 2.0 ** -53
    err = np.linalg.norm(v.reshape(-1) - full[:, 0])
    # sums of r products per core, relative to the product of the cores' norms (largest singular value times sqrt(r))
    scale = np.prod([np.linalg.norm(a.astype(np.complex128)) / (r ** 0.5 if k else 1) for k, a in enumerate(x)])
    assert err <= 20 * len(modes) * max(r, 2) ** 0.5 * u * max(np.linalg.norm(full), scale)
