"""GPU: the direct split (Householder bidiagonalisation, divide and conquer on
the FP64 tridiagonal, blocked back-transformation) against numpy's SVD of the
same weighted matrix, at the edges of its kernels: leaf sizes (8), reflector
panels (32), one CTA per problem / few CTAs / many CTAs, tall, square and wide
matrices, several problems of different width in one step, rank-deficient and
exactly degenerate inputs, in both precisions.

Tolerances: Householder transformations and the products around them have a
backward error of about eps sqrt(n) |M| with a small constant; 8 eps sqrt(n)
bounds theta and the isometry, and f is second order in the subspace."""
import numpy as np
import pytest

from gpu_helpers import lib

pytestmark = pytest.mark.gpu
EPS = {"FP32": 2.0 ** -23, "FP64": 2.0 ** -52}


def _site(rng, a, b):
    """Random tensor with orthonormal rows where a <= 2 b, else normalised."""
    g = rng.standard_normal((a, 2 * b)) + 1j * rng.standard_normal((a, 2 * b))
    if a <= 2 * b:
        g = np.linalg.qr(g.conj().T)[0].conj().T
    return g.reshape(a, 2, b) if a <= 2 * b else (g / np.linalg.norm(g)).reshape(a, 2, b)


def _state(rng, shapes, dtype, decades=4.0):
    """Sites of two-site blocks (a, b, c) side by side, joined by bonds of 1."""
    chis, sites = [1], []
    for a, b, c in shapes:
        for x, y in ((1, a), (a, b), (b, c), (c, 1)):
            sites.append(_site(rng, x, y).astype(dtype))
            chis.append(y)
    lams = []
    for c in chis:
        w = np.sort(rng.exponential(1.0, c) * 10.0 ** (-decades * np.arange(c) / c))[::-1]
        lams.append(np.sqrt(w / w.sum()))
    return np.array(chis, dtype=np.int32), sites, lams


def _check(P, chis, sites, lams, q0s, Us, prec, chi_max, cutoff):
    n = len(sites)
    lg = int(np.ceil(np.log2(max(chi_max, max(chis), 2))))
    cfg = P.make_config(n, max(chi_max, int(max(chis))), cutoff, 4 + 2 * lg, 0, 2, getattr(P, prec))
    mps = P.MPS(cfg)
    mps.load(chis, sites, lams)
    fs = mps.step([P.Cluster(q, 2, 0, 0) for q in q0s], Us)
    assert np.all(mps.split_log()[:, 12:14] == 0)   # no Jacobi sweeps: the direct solver ran
    eps = EPS[prec]
    floor = 1e-13 if prec == "FP64" else 1e-6
    for q0, U, f in zip(q0s, Us, fs):
        a, c = int(chis[q0]), int(chis[q0 + 2])
        A, B = sites[q0].astype(np.complex128), sites[q0 + 1].astype(np.complex128)
        th = np.einsum("st,atb->asb", U, np.tensordot(A, B, axes=([2], [0])).reshape(a, 4, c))
        M = np.repeat(lams[q0], 2)[:, None] * th.reshape(2 * a, 2 * c)
        u, s, vh = np.linalg.svd(M, full_matrices=False)
        p = s * s
        tail = np.append(np.cumsum(p[::-1])[::-1][1:], 0.0)
        r = int(np.argmax(tail <= cutoff * p.sum())) + 1 if cutoff > 0 else len(p)
        r = max(1, min(r, int((p > floor ** 2 * p[0]).sum()), cfg.chi_max))
        got = int(mps.bond_dims()[q0 + 1])
        assert got == r, (a, c, got, r)
        tol = 8 * eps * np.sqrt(max(M.shape))
        left = mps.site(q0).astype(np.complex128)
        right = mps.site(q0 + 1).astype(np.complex128).reshape(r, 2 * c)
        assert np.max(np.abs(right @ right.conj().T - np.eye(r))) <= tol
        want = (u[:, :r] * s[:r]) @ vh[:r] / np.sqrt(p[:r].sum())
        have = (lams[q0][:, None] * left.reshape(a, -1)).reshape(2 * a, r) @ right
        # the kept subspace turns by noise / gap at the cut: compare its weight there, and theta
        # where nothing but numerical zeros is dropped
        if r == min(M.shape) or p[min(r, len(p) - 1)] <= 1e-3 * p[r - 1]:
            assert np.linalg.norm(have - want) <= tol * np.linalg.norm(want), (a, c)
        assert abs(f - p[:r].sum() / p.sum()) <= max(tol, 4 * eps)
        np.testing.assert_allclose(mps.lam(q0 + 1), s[:r] / np.sqrt(p[:r].sum()), rtol=0, atol=tol)


def _unitary(rng):
    return np.linalg.qr(rng.standard_normal((4, 4)) + 1j * rng.standard_normal((4, 4)))[0]


# (chi_L, chi_mid, chi_R): the split matrix is 2 chi_L x 2 chi_R
SHAPES = [(1, 1, 1), (1, 2, 4), (2, 4, 4), (4, 5, 5), (5, 9, 16), (16, 16, 17), (32, 32, 32), (33, 40, 33),
          (64, 64, 64), (65, 70, 65), (128, 128, 31), (31, 62, 100), (100, 128, 128), (129, 129, 129),
          (300, 310, 290)]


@pytest.mark.parametrize("prec", ["FP32", "FP64"])
@pytest.mark.parametrize("shape", SHAPES)
def test_direct_split_shapes(shape, prec):
    rng = np.random.default_rng(sum(shape))
    chis, sites, lams = _state(rng, [shape], np.complex64 if prec == "FP32" else np.complex128)
    cap = 2 * max(shape)
    _check(lib(), chis, sites, lams, [1], [_unitary(rng)], prec, cap, 0.0)
    _check(lib(), chis, sites, lams, [1], [_unitary(rng)], prec, max(1, min(shape) // 2), 0.0)


@pytest.mark.parametrize("prec", ["FP32", "FP64"])
def test_direct_split_mixed_widths(prec):
    """One step over problems of very different widths (several launch classes)."""
    rng = np.random.default_rng(3)
    shapes = [(3, 5, 6), (40, 40, 44), (1, 2, 2), (90, 100, 96), (64, 64, 64), (12, 20, 150), (7, 7, 7)]
    chis, sites, lams = _state(rng, shapes, np.complex64 if prec == "FP32" else np.complex128)
    _check(lib(), chis, sites, lams, [1 + 4 * i for i in range(len(shapes))], [_unitary(rng) for _ in shapes], prec, 300, 0.0)


@pytest.mark.parametrize("prec", ["FP32", "FP64"])
@pytest.mark.parametrize("rank", [1, 3, 20])
def test_direct_split_rank_deficient(rank, prec):
    """theta of low rank with a flat, exactly degenerate spectrum: only the rank survives."""
    rng = np.random.default_rng(rank)
    chis, sites, lams = _state(rng, [(40, rank, 40)], np.complex64 if prec == "FP32" else np.complex128)
    lams[1] = np.full(40, 1 / np.sqrt(40))
    _check(lib(), chis, sites, lams, [1], [np.eye(4, dtype=np.complex128)], prec, 80, 0.0)


@pytest.mark.parametrize("prec", ["FP32", "FP64"])
@pytest.mark.parametrize("decades", [8.0, 16.0])
def test_direct_split_steep_wide(decades, prec):
    """Fewer rows than columns and a steep spectrum: behind the rank, the bidiagonal ends in rounding
    noise whose squares lie below FP32's range."""
    rng = np.random.default_rng(int(decades))
    chis, sites, lams = _state(rng, [(96, 98, 100)], np.complex64 if prec == "FP32" else np.complex128, decades)
    _check(lib(), chis, sites, lams, [1], [_unitary(rng)], prec, 200, 1e-9)


def test_direct_split_larger_than_shared_memory():
    """FP32 rows that do not fit the chip's shared memory (m = 4 n through a three-site cluster)."""
    P = lib()
    rng = np.random.default_rng(11)
    chi = 640
    chis, sites, lams = _state(rng, [(2 * chi, 2 * chi, chi)], np.complex64)
    cfg = P.make_config(len(sites), 2 * chi, 0.0, 3 + 2 * 11, 0, 2, P.FP32)
    mps = P.MPS(cfg)
    mps.load(chis, sites, lams)
    f = mps.step([P.Cluster(1, 2, 0, 0)], [np.eye(4, dtype=np.complex128)])
    assert abs(f[0] - 1) <= 8 * EPS["FP32"] * np.sqrt(4 * chi)
    r = int(mps.bond_dims()[2])
    right = mps.site(2).astype(np.complex128).reshape(r, -1)
    assert np.max(np.abs(right @ right.conj().T - np.eye(r))) <= 8 * EPS["FP32"] * np.sqrt(4 * chi)
