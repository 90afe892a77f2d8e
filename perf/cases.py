"""Workloads that a user of the library has it do, for timing and for comparing
results: TT rounding (SVD and sketched, one train and a batch), the contrast
and SFFT steps of the Moulinec-Suquet iteration, inner products, TT-SVD of a
phase image, and whole homogenisation solves, in complex64 and complex128.

Trains that a rounding returns have cores that are unique only up to a gauge, so
those passes end with contract() (tt_contract_voxels), which returns the whole
tensor.  Bond indices of the drawn trains carry weights that fall over some six
decades, as the singular values of the strain iterates do."""
import math

import numpy as np
import torch

from paper_2512_07811_gb300 import inputs as I
from paper_2512_07811_gb300 import qtt as Q

_CTX = []


def _ctx():
    # one context per process, as a program opens it
    if not _CTX:
        _CTX.append(Q.Context(0))
    return _CTX[0]


def listed():
    return [
        # the smallest sum-and-round: a 16^3 grid's train at rank 16 (launches and latency count)
        {"name": "add_round_c64_d12_r16", "op": "add_round", "dtype": "c64", "d": 12, "r": 16, "eps": 1e-6},
        # x + y rounded at the ordinary rank of the TT-op sweep, on a 64^3 grid's 18 sites
        {"name": "add_round_c64_d18_r64", "op": "add_round", "dtype": "c64", "d": 18, "r": 64, "eps": 1e-6},
        # the largest SVD rounding: bonds of 192 rounded on 20 sites
        {"name": "add_round_c64_d20_r96", "op": "add_round", "dtype": "c64", "d": 20, "r": 96, "eps": 1e-6},
        # the same operation on the FP64 path, at an odd rank
        {"name": "add_round_c128_d14_r37", "op": "add_round", "dtype": "c128", "d": 14, "r": 37, "eps": 1e-9},
        # many trains of one shape rounded together (load cases, RVEs)
        {"name": "round_batch_c64_d14_r32_x12", "op": "round_batch", "dtype": "c64", "d": 14, "r": 32, "count": 12,
         "eps": 1e-6},
        # the contrast step of an elastic 32^3 solve at the headline's ranks (cap 128, sketch
        # width 136, phase train 113): round(a eps + b chi eps), control core of 6 components
        {"name": "contrast_c64_d15_r128", "op": "contrast", "dtype": "c64", "d": 15, "r": 128, "chi": 113, "ncomp": 6,
         "eps": 1e-6},
        # the same step of a small scalar problem on the FP64 path
        {"name": "contrast_c128_d12_r40", "op": "contrast", "dtype": "c128", "d": 12, "r": 40, "chi": 12, "ncomp": 3,
         "eps": 1e-9},
        # the SFFT step: Q_n x rounded, rank of the TT-op sweep
        {"name": "sfft_c64_d16_r64", "op": "sfft", "dtype": "c64", "d": 16, "r": 64, "eps": 1e-6},
        # inner product and norm of long trains (stop test, effective tensor)
        {"name": "dot_norm_c64_d30_r128", "op": "dot_norm", "dtype": "c64", "d": 30, "r": 128},
        # operator setup: TT-SVD of a 32^3 phase image
        {"name": "from_dense_c128_32", "op": "from_dense", "dtype": "c128", "d": 15, "eps": 1e-10},
        # whole solve, float path: elastic sphere, six load cases on their own streams
        {"name": "ms_elastic_c64_16", "op": "ms", "dtype": "c64", "kind": "elastic", "n": 4, "iters": 4, "r": 128,
         "eps": 1e-6, "op_tol": 1e-6, "contrast": 10.0},
        # whole solve, FP64 path: the scalar 32^3 laminate
        {"name": "ms_laminate_c128_32", "op": "ms", "dtype": "c128", "kind": "laminate", "n": 5, "iters": 2, "r": 64,
         "eps": 1e-9, "op_tol": 1e-11, "contrast": 10.0},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["add_round", "add_round", "add_round", "round_batch", "contrast", "contrast", "sfft", "dot_norm",
                     "from_dense", "ms"])
    dt = rng.choice(["c64", "c64", "c128"])
    eps = 1e-6 if dt == "c64" else 1e-9
    if op == "add_round":
        return {"op": op, "dtype": dt, "d": rng.randint(10, 20 if dt == "c64" else 14),
                "r": _log_int(rng, 9, 96 if dt == "c64" else 40), "eps": eps}
    if op == "round_batch":
        return {"op": op, "dtype": dt, "d": rng.randint(10, 14), "r": _log_int(rng, 8, 48 if dt == "c64" else 20),
                "count": rng.randint(2, 12), "eps": eps}
    if op == "contrast":
        return {"op": op, "dtype": dt, "d": rng.randint(9, 15 if dt == "c64" else 12),
                "r": _log_int(rng, 20, 128 if dt == "c64" else 40), "chi": _log_int(rng, 6, 113 if dt == "c64" else 16),
                "ncomp": rng.choice([3, 6]), "eps": eps}
    if op == "sfft":
        return {"op": op, "dtype": dt, "d": rng.randint(10, 16 if dt == "c64" else 13),
                "r": _log_int(rng, 12, 64 if dt == "c64" else 32), "eps": eps}
    if op == "dot_norm":
        return {"op": op, "dtype": dt, "d": rng.randint(10, 30), "r": _log_int(rng, 8, 128 if dt == "c64" else 40)}
    if op == "from_dense":
        return {"op": op, "dtype": "c128", "d": rng.choice([9, 12, 15]), "eps": 1e-10}
    if dt == "c64":
        return {"op": op, "dtype": dt, "kind": "elastic", "n": rng.choice([3, 4]), "iters": rng.randint(2, 4), "r": 128,
                "eps": 1e-6, "op_tol": 1e-6, "contrast": round(math.exp(rng.uniform(math.log(5), math.log(20))), 3)}
    return {"op": op, "dtype": dt, "kind": "laminate", "n": rng.choice([3, 4, 5]), "iters": rng.randint(1, 2),
            "r": rng.choice([32, 64]), "eps": 1e-9, "op_tol": 1e-11,
            "contrast": round(math.exp(rng.uniform(math.log(2), math.log(20))), 3)}


# ------------------------------------------------------------------ inputs

def _dt(case):
    return Q.C64 if case["dtype"] == "c64" else Q.C128


def _np(case):
    return np.complex64 if case["dtype"] == "c64" else np.complex128


def _ranks(modes, r):
    out = [1]
    for k in range(1, len(modes)):
        out.append(int(min(r, math.prod(modes[:k]), math.prod(modes[k:]))))
    return out + [1]


def _train(rng, modes, r, case, decades=None):
    """Gaussian cores whose right bond indices carry weights falling over `decades` decades
    (six in complex64, nine in complex128: the rounding tolerance), values of the case's dtype."""
    if decades is None:
        decades = 6.0 if case["dtype"] == "c64" else 9.0
    ranks = _ranks(modes, r)
    cores = []
    for k, n in enumerate(modes):
        a = rng.standard_normal((ranks[k], n, ranks[k + 1])) + 1j * rng.standard_normal((ranks[k], n, ranks[k + 1]))
        m = ranks[k + 1]
        a *= 10.0 ** (-decades * np.arange(m) / max(r, 1))
        cores.append((a / math.sqrt(2.0 * n * max(1.0, 0.1 * ranks[k]))).astype(_np(case)))
    return cores


def _grid(d):
    return [(d + 2) // 3, (d + 1) // 3, d // 3]


def _sphere(rng):
    centre = rng.uniform(0.3, 0.7, 3)
    return I.sphere_rows(float(rng.uniform(0.17, 0.23)), tuple(centre))


def _image_sites(case, rng):
    """Phase image of a sphere on a 2^(d/3) grid, as the tensor of its bit-interleaved sites."""
    n = case["d"] // 3
    N = 1 << n
    img = I.ellipsoids_indicator(_sphere(rng), (N, N, N))
    axes = [a * n + p for p in range(n) for a in range(3)]
    return np.ascontiguousarray(img.reshape((2,) * (3 * n)).transpose(axes)).reshape(-1)


def _ms_problem(case, rng):
    N = 1 << case["n"]
    if case["kind"] == "laminate":
        img = I.laminate_indicator(N, axis=0, fraction=float(rng.choice([0.25, 0.5, 0.75])))
        k1, k2 = 1.0, float(case["contrast"] * rng.uniform(0.9, 1.1))
        return img, img, "scalar", (k1, k2), 0.5 * (k1 + k2) * np.eye(3), True
    rows = _sphere(rng)
    l1, m1 = I.lame_from_young(1.0, 0.3)
    l2, m2 = I.lame_from_young(float(case["contrast"] * rng.uniform(0.9, 1.1)), 0.3)
    return (Q.Ellipsoids(rows, (N, N, N)), I.ellipsoids_indicator(rows, (N, N, N)), "elastic", (l1, m1, l2, m2),
            _voigt(0.5 * (l1 + l2), 0.5 * (m1 + m2)), False)


def _voigt(lam, mu):
    C = np.zeros((6, 6))
    C[:3, :3] = lam
    C[range(3), range(3)] += 2 * mu
    C[range(3, 6), range(3, 6)] = mu
    return C


def _data(case, seed):
    """The host-side inputs of a case, from the seed alone."""
    rng = np.random.default_rng([int(seed), 20251207])
    op = case["op"]
    if op == "add_round":
        modes = [2] * case["d"]
        return {"x": _train(rng, modes, case["r"], case), "y": _train(rng, modes, case["r"], case), "a": 1.0, "b": 0.5}
    if op == "round_batch":
        modes = [2] * case["d"]
        return {"x": [_train(rng, modes, 2 * case["r"], case) for _ in range(case["count"])]}
    if op == "contrast":
        modes = [case["ncomp"]] + [2] * case["d"]
        return {"x": _train(rng, modes, case["r"], case), "chi": _train(rng, modes, case["chi"], case, 3.0),
                "a": -0.45, "b": 0.9, "sketch": I.sketch_cores(rng, len(modes), modes, case["r"] + 8)[0]}
    if op == "sfft":
        modes = [2] * case["d"]
        return {"x": _train(rng, modes, case["r"], case), "sketch": I.sketch_cores(rng, len(modes), modes,
                                                                                     case["r"] + 8)[0]}
    if op == "dot_norm":
        x = _train(rng, [2] * case["d"], case["r"], case, 3.0)
        y = [(c * (1.0 + 0.2 * rng.standard_normal(c.shape))).astype(_np(case)) for c in x]
        return {"x": x, "y": y}
    if op == "from_dense":
        return {"dense": _image_sites(case, rng)}
    if op == "ms":
        return {"problem": _ms_problem(case, rng)}
    raise ValueError(op)


def prepare(case, seed):
    ctx, dt, h = _ctx(), _dt(case), _data(case, seed)
    s = {"case": case, "ctx": ctx}
    op = case["op"]
    tt = lambda cores: Q.TT.from_cores(ctx, cores, dt)  # noqa: E731
    if op == "add_round":
        s.update(x=tt(h["x"]), y=tt(h["y"]), a=h["a"], b=h["b"])
    elif op == "round_batch":
        s.update(x=[tt(x) for x in h["x"]])
    elif op == "contrast":
        s.update(x=tt(h["x"]), chi=Q.qtt_mpo_diag(ctx, tt(h["chi"])), a=h["a"], b=h["b"], sketch=tt(h["sketch"]))
    elif op == "sfft":
        F = Q.qtt_qft_mpo(ctx, case["d"], -1, 1e-12)
        s.update(x=tt(h["x"]), sketch=tt(h["sketch"]), F=F if dt == Q.C128 else Q.qtt_mpo_convert(ctx, F, dt))
    elif op == "dot_norm":
        s.update(x=tt(h["x"]), y=tt(h["y"]))
    elif op == "from_dense":
        s.update(dense=torch.from_numpy(h["dense"].astype(np.complex128)).cuda())
    elif op == "ms":
        geo, _, kind, moduli, C0, inter = h["problem"]
        s.update(kind=kind, moduli=moduli, C0=C0, geo=geo, inter=inter,
                 ops=Q.ms_setup(ctx, geo, kind, moduli, C0, op_tol=case["op_tol"], interleaved=inter,
                                op_prec=Q.PREC_F32 if dt == Q.C64 else Q.PREC_F64))
    ctx.sync()
    return s


# ------------------------------------------------------------------- a pass

def run(s):
    case, ctx = s["case"], s["ctx"]
    op = case["op"]
    if op == "add_round":
        z = Q.tt_add(ctx, s["a"], s["x"], s["b"], s["y"])
        y, _ = Q.tt_round(ctx, z, case["eps"])
        return Q.contract_voxels(ctx, y, _grid(case["d"]))
    if op == "round_batch":
        ys, _ = Q.tt_round_batch(ctx, s["x"], case["eps"])
        return [Q.contract_voxels(ctx, y, _grid(case["d"])) for y in ys]
    if op == "contrast":
        y, _ = Q.tt_round_sketched(ctx, [(s["a"], None, s["x"]), (s["b"], s["chi"], s["x"])], s["sketch"], case["eps"],
                                   case["r"])
        return Q.contract_voxels(ctx, y, _grid(case["d"]))
    if op == "sfft":
        y, _ = Q.tt_round_sketched(ctx, [(1.0, s["F"], s["x"])], s["sketch"], case["eps"], case["r"])
        return Q.contract_voxels(ctx, y, _grid(case["d"]))
    if op == "dot_norm":
        # the values carry the precision of the trains they were computed in
        real = np.float32 if case["dtype"] == "c64" else np.float64
        return [_np(case)(Q.tt_dot(ctx, s["x"], s["y"])), real(Q.tt_norm(ctx, s["x"]))]
    if op == "from_dense":
        y = Q.tt_from_dense(ctx, s["dense"].data_ptr(), [2] * case["d"], case["eps"])
        return Q.contract_voxels(ctx, y, _grid(case["d"]))
    if op == "ms":
        C, rep = Q.ms_homogenize(ctx, s["geo"], s["kind"], s["moduli"], s["C0"], tol=0.0, max_rank=case["r"],
                               eps=case["eps"], op_tol=case["op_tol"], max_iter=case["iters"], min_iter=case["iters"],
                               prec=Q.PREC_F32 if case["dtype"] == "c64" else Q.PREC_F64, interleaved=s["inter"],
                               lc_workers=6 if s["kind"] == "elastic" else 1, ops=s["ops"],
                               return_strain=case["dtype"] == "c128")
        if case["dtype"] == "c64":
            return C.astype(np.float32)  # the float path computes C_eff in single precision
        return [C, Q.contract_voxels(ctx, rep.strain, [case["n"]] * 3, s["inter"])]
    raise ValueError(op)


# --------------------------------------------------------- what it has to do

def _qr_flops(m, n):
    k = min(m, n)
    return 8.0 * (2.0 * m * n * k - (m + n) * k * k + 2.0 * k ** 3 / 3.0)


def _round_work(modes, r_in, r_out, el, left_orth=False):
    """One SVD rounding: QR sweep (absorb R, R factors), truncated-SVD sweep, cores once in and out."""
    d = len(modes)
    R = [1] * (d + 1)
    f = 0.0
    for k in range(d - 1):
        R[k + 1] = min(R[k] * modes[k], r_in[k + 1])
        if not left_orth:
            f += 8.0 * R[k] * r_in[k] * modes[k] * r_in[k + 1] + _qr_flops(R[k] * modes[k], r_in[k + 1])
    for k in range(d - 1, 0, -1):
        p, q = modes[k] * r_out[k + 1], R[k]
        mn = min(p, q)
        f += 16.0 * max(p, q) * mn * mn + 32.0 * mn ** 3 + 8.0 * modes[k - 1] * r_in[k - 1] * r_in[k] * r_out[k]
    by = sum(a * n * b for a, n, b in zip(r_in, modes, r_in[1:])) + sum(a * n * b
                                                                        for a, n, b in zip(r_out, modes, r_out[1:]))
    return f, by * el


def _sketch_work(modes, terms, ell, el):
    """Right partial contractions of the structured sum with the sketch, and the left-to-right projection;
    terms: (operator ranks, train ranks), diagonal or 2x2 operator cores counted as stored nonzeros."""
    d = len(modes)
    f = by = 0.0
    for g, r, diag in terms:
        for k in range(d):
            n = modes[k]
            nn = n if diag else n * n
            lr = 8.0 * (g[k + 1] * r[k + 1] * n * ell[k] * ell[k + 1] + nn * g[k] * g[k + 1] * r[k + 1] * ell[k] +
                        g[k] * r[k] * n * r[k + 1] * ell[k])
            f += 2.0 * lr
            by += (r[k] * n * r[k + 1] + nn * g[k] * g[k + 1]) * el
    for k in range(d - 1):
        f += 2.0 * _qr_flops(ell[k] * modes[k], ell[k + 1])
    by += sum(a * n * b for a, n, b in zip(ell, modes, ell[1:])) * el
    return f, by


def work(case):
    el = 8 if case["dtype"] == "c64" else 16
    op = case["op"]
    if op in ("add_round", "round_batch"):
        modes = [2] * case["d"]
        r1, r2 = _ranks(modes, case["r"]), _ranks(modes, 2 * case["r"])
        f, by = _round_work(modes, [1] + [2 * v for v in r1[1:-1]] + [1] if op == "add_round" else r2, r2, el)
        f += 8.0 * sum(2.0 ** (k + 1) * r2[k] * r2[k + 1] for k in range(len(modes)))
        by += 2.0 ** case["d"] * el
        c = case.get("count", 1)
        return {"bytes": c * by, "flops": c * f}
    if op in ("contrast", "sfft"):
        modes = ([case["ncomp"]] if op == "contrast" else []) + [2] * case["d"]
        r, ell = _ranks(modes, case["r"]), _ranks(modes, case["r"] + 8)
        one = [1] * (len(modes) + 1)
        if op == "contrast":
            terms = [(one, r, True), (_ranks(modes, case["chi"]), r, True)]
        else:
            terms = [(_ranks([4] * case["d"], 8), r, False)]
        f, by = _sketch_work(modes, terms, ell, el)
        f2, _ = _round_work(modes, ell, r, el, left_orth=True)
        n = math.prod(modes)
        return {"bytes": by + n * el, "flops": f + f2 + 8.0 * sum(2.0 ** (k + 1) * r[k] * r[k + 1]
                                                                 for k in range(len(modes)))}
    if op == "dot_norm":
        modes = [2] * case["d"]
        r = _ranks(modes, case["r"])
        f = sum(16.0 * r[k] * 2 * r[k + 1] * (r[k] + r[k + 1]) / 2 * 1.0 for k in range(case["d"]))
        f += sum(8.0 * r[k] * r[k] * 2 * r[k + 1] + _qr_flops(2 * r[k], r[k + 1]) for k in range(case["d"]))
        return {"bytes": 2.0 * el * sum(a * 2 * b for a, b in zip(r, r[1:])), "flops": f}
    if op == "from_dense":
        # one SVD per unfolding, at the ranks that a sphere's phase image has (about 2.5 x per doubled grid)
        d = case["d"]
        r = [1] + [int(min(2 ** k, 2 ** (d - k), 72 * 2.5 ** (d / 3 - 5))) for k in range(1, d)] + [1]
        f = sum(16.0 * 2.0 ** (d - k - 1) * (2 * r[k]) ** 2 + 8.0 * r[k + 1] * 2 * r[k] * 2.0 ** (d - k - 1)
                for k in range(d - 1))
        return {"bytes": 2.0 * el * 2 ** d, "flops": f}
    # the four roundings of every iteration and load case at the ranks that the grid allows
    nc = 6 if case["kind"] == "elastic" else 3
    modes = [nc] + [2] * (3 * case["n"])
    r, ell = _ranks(modes, case["r"]), _ranks(modes, case["r"] + 8)
    g = _ranks([nc * nc] + [2] * (3 * case["n"]), 125 if nc == 6 else 30)
    f1, b1 = _sketch_work(modes, [(g, r, True)], ell, el)
    f2, _ = _round_work(modes, ell, r, el, left_orth=True)
    m = case["iters"] * nc
    return {"bytes": m * 2.0 * b1, "flops": m * (f1 + 4.0 * f2)}


# ------------------------------------------------- the same in plain 64 bits

def _z(cores):
    return [torch.from_numpy(np.ascontiguousarray(c)).to(torch.complex128).cuda() for c in cores]


def _full(cores):
    t = cores[0].reshape(-1, cores[0].shape[2])
    for c in cores[1:]:
        t = (t @ c.reshape(c.shape[0], -1)).reshape(-1, c.shape[2])
    return t.reshape(-1)


def _tt_round_full(t, modes, eps, cap=0):
    """SVD rounding of a whole tensor, from the last bond to the first, threshold eps ||t|| / sqrt(d - 1)."""
    d = len(modes)
    delta = eps * float(torch.linalg.vector_norm(t)) / math.sqrt(d - 1)
    cores, r = [], 1
    for k in range(d - 1, 0, -1):
        m = t.reshape(-1, modes[k] * r)
        if m.shape[0] > m.shape[1]:
            # right vectors of the triangular factor are those of m
            vh, s = torch.linalg.svd(torch.linalg.qr(m, mode="r")[1], full_matrices=False)[2], None
            s = torch.linalg.vector_norm(m @ vh.mH, dim=0)
        else:
            _, s, vh = torch.linalg.svd(m, full_matrices=False)
        tail = torch.sqrt(torch.flip(torch.cumsum(torch.flip(s * s, [0]), 0), [0]))
        keep = max(1, int((tail > delta).sum()))
        keep = min(keep, cap) if cap else keep
        vh = vh[:keep]
        cores.insert(0, vh.reshape(keep, modes[k], r))
        t, r = m @ vh.mH, keep
    cores.insert(0, t.reshape(1, modes[0], r))
    return _full(cores)


def _project(t, modes, sketch):
    """Left-to-right projection of a whole tensor on the ranges of its sketched unfoldings."""
    d = len(modes)
    right = [None] * (d + 1)
    right[d] = torch.ones(1, 1, dtype=torch.complex128, device=t.device)
    for k in range(d - 1, 0, -1):
        c = sketch[k]
        right[k] = (c.reshape(-1, c.shape[2]) @ right[k + 1]).reshape(c.shape[0], -1)
    cores, l = [], 1
    for k in range(d - 1):
        m = t.reshape(l * modes[k], -1)
        q = torch.linalg.qr(m @ right[k + 1].T)[0]
        cores.append(q.reshape(l, modes[k], -1))
        t, l = q.mH @ m, q.shape[1]
    cores.append(t.reshape(l, modes[-1], 1))
    return _full(cores)


def _voxels(t, ncomp, nbits):
    """Site order (control first, then bit-interleaved sites) to a voxel field."""
    sites = []
    for p in range(max(nbits)):
        sites += [(a, p) for a in range(3) if p < nbits[a]]
    order = [1 + sites.index((a, p)) for a in range(3) for p in range(nbits[a])]
    t = t.reshape([ncomp] + [2] * len(sites)).permute([0] + order)
    return t.reshape([ncomp] + [1 << b for b in nbits]).contiguous().cpu().numpy()


def _ms_exact(case, h):
    _, img, kind, moduli, C0, _ = h["problem"]
    nc = C0.shape[0]
    if kind == "scalar":
        C1, C2 = moduli[0] * np.eye(3), moduli[1] * np.eye(3)
    else:
        C1, C2 = _voigt(*moduli[:2]), _voigt(*moduli[2:])
    N = img.shape[0]
    k = np.fft.fftfreq(N) * N
    xi = np.stack(np.meshgrid(k, k, k, indexing="ij"))
    q2 = (xi ** 2).sum(0)
    q2[0, 0, 0] = 1.0
    if kind == "scalar":
        G = xi[:, None] * xi[None] / (C0[0, 0] * q2)
    else:
        lam, mu = C0[0, 1], C0[3, 3]
        pairs, w = [(0, 0), (1, 1), (2, 2), (1, 2), (0, 2), (0, 1)], [1, 1, 1, 2, 2, 2]
        G = np.zeros((6, 6) + img.shape)
        for a, (i, j) in enumerate(pairs):
            for b, (p, q) in enumerate(pairs):
                g = ((p == i) * xi[q] * xi[j] + (q == i) * xi[p] * xi[j] + (p == j) * xi[q] * xi[i] +
                     (q == j) * xi[p] * xi[i]) / (4 * mu * q2)
                g = g - (lam + mu) / (mu * (lam + 2 * mu)) * xi[i] * xi[j] * xi[p] * xi[q] / q2 ** 2
                G[a, b] = w[a] * w[b] * g
    G[:, :, 0, 0, 0] = 0.0
    to = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(torch.complex128).cuda()  # noqa: E731
    G, chi, A, B, C1, D = to(G), to(img), to(C1 - C0), to(C2 - C1), to(C1), to(C2 - C1)
    out = np.zeros((nc, nc))
    for c in range(nc):
        E = torch.zeros(nc, 1, 1, 1, dtype=torch.complex128, device="cuda")
        E[c] = 1.0
        e = E.expand(nc, N, N, N)
        for _ in range(case["iters"]):
            tau = torch.einsum("ij,jxyz->ixyz", A, e) + chi * torch.einsum("ij,jxyz->ixyz", B, e)
            e = E - torch.fft.ifftn(torch.einsum("ijxyz,jxyz->ixyz", G, torch.fft.fftn(tau, dim=(1, 2, 3))),
                                    dim=(1, 2, 3))
        sig = torch.einsum("ij,jxyz->ixyz", C1, e) + chi * torch.einsum("ij,jxyz->ixyz", D, e)
        out[:, c] = sig.mean(dim=(1, 2, 3)).real.cpu().numpy()
    return out if case["dtype"] == "c64" else [out, e.contiguous().cpu().numpy()]


def exact(case, seed):
    h, op = _data(case, seed), case["op"]
    if op == "ms":
        return _ms_exact(case, h)
    if op == "dot_norm":
        x, y = _z(h["x"]), _z(h["y"])

        def inner(u, v):
            w = torch.ones(1, 1, dtype=torch.complex128, device="cuda")
            for a, b in zip(u, v):
                w = torch.einsum("ab,anc,bnd->cd", w, a.conj(), b)
            return complex(w.item())

        return [np.complex128(inner(x, y)), np.float64(math.sqrt(inner(x, x).real))]
    if op == "from_dense":
        return _voxels(torch.from_numpy(h["dense"].astype(np.complex128)), 1, _grid(case["d"]))
    nbits = _grid(case["d"])
    modes = [2] * case["d"]
    if op == "add_round":
        t = h["a"] * _full(_z(h["x"])) + h["b"] * _full(_z(h["y"]))
        return _voxels(_tt_round_full(t, modes, case["eps"]), 1, nbits)
    if op == "round_batch":
        return [_voxels(_tt_round_full(_full(_z(x)), modes, case["eps"]), 1, nbits) for x in h["x"]]
    x, sk = _full(_z(h["x"])), _z([c.astype(_np(case)) for c in h["sketch"]])
    if op == "contrast":
        modes = [case["ncomp"]] + modes
        t, nc = h["a"] * x + h["b"] * _full(_z(h["chi"])) * x, case["ncomp"]
    else:
        d = case["d"]
        t = torch.fft.fft(x, norm="ortho").reshape([2] * d).permute(list(range(d))[::-1]).reshape(-1)
        nc = 1
    t = _tt_round_full(_project(t, modes, sk), modes, case["eps"], case["r"])
    return _voxels(t, nc, nbits)
