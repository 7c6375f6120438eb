"""GPU: all splits of a narrow cluster in one launch (Householder QR, one-sided
Jacobi, truncation in one CTA) against numpy's SVDs of the same matrices, at
the edges of the kernel: one to 16 columns, fewer rows than columns, odd sizes,
more rows than threads, the widths on both sides of its limit, two to six
sites, truncated and not, rank-deficient, in both precisions.

Tolerances: the arithmetic is FP64 in both precisions and the results are
rounded to the tensors' type once per split; every split before it moves the
remainder by the same, so 8 eps k sqrt(elements of a row) bounds theta, the
isometries and the spectra, and f is second order in the subspace."""
import numpy as np
import pytest

from gpu_helpers import lib

pytestmark = pytest.mark.gpu
EPS = {"FP32": 2.0 ** -23, "FP64": 2.0 ** -52}


def _splits(M, lam, k, chi_max, floor):
    """numpy: the k - 1 splits of M (chi_L x 2^k x chi_R), right to left -> (spectra, fidelity, theta kept)."""
    chiL, chiR = M.shape[0], M.shape[2]
    cur, rdim, f, spectra, V = M.reshape(chiL, -1), chiR, 1.0, {}, None
    for j in range(k - 1, 0, -1):
        mat = (np.repeat(lam, 2 ** j)[:, None] * cur.reshape(chiL * 2 ** j, 2 * rdim))
        u, s, vh = np.linalg.svd(mat, full_matrices=False)
        p = s * s
        r = max(1, min(int((p > floor ** 2 * p[0]).sum()), chi_max))
        f *= p[:r].sum() / p.sum()
        kept = np.sqrt(p[:r].sum())
        spectra[j] = s[:r] / kept
        cur, rdim = (cur.reshape(chiL * 2 ** j, -1) @ vh[:r].conj().T) / kept, r
        tail = vh[:r].reshape(r, 2, -1)
        V = tail if V is None else np.tensordot(tail, V, axes=([2], [0]))
    return spectra, f, lam[:, None] * np.tensordot(cur.reshape(chiL * 2, rdim), V.reshape(rdim, -1), 1).reshape(chiL, -1)


def _check(P, chiL, chiR, k, prec, inner=None):
    chi_max = 600
    rng = np.random.default_rng(100 * chiL + 10 * chiR + k)
    dtype = np.complex64 if prec == "FP32" else np.complex128
    chis = [1, chiL]
    for j in range(1, k):
        chis.append(min(inner or 64, chis[-1] * 2, chiR * 2 ** (k - j)))
    chis += [chiR, 1]
    sites = []
    for a, b in zip(chis[:-1], chis[1:]):
        g = rng.standard_normal((a, 2 * b)) + 1j * rng.standard_normal((a, 2 * b))
        sites.append((g / np.linalg.norm(g)).reshape(a, 2, b).astype(dtype))
    lams = [np.sort(rng.random(c) + 0.05)[::-1] for c in chis]
    lams = [l / np.linalg.norm(l) for l in lams]
    d = 2 ** k
    U = np.linalg.qr(rng.standard_normal((d, d)) + 1j * rng.standard_normal((d, d)))[0] if not inner else np.eye(d) + 0j
    cfg = P.make_config(k + 2, chi_max, 0.0, 2 * k + 24, 0, k, getattr(P, prec))
    mps = P.MPS(cfg)
    mps.load(np.array(chis, dtype=np.int32), sites, lams)
    f = np.prod(mps.step([P.Cluster(1, k, 0, 0)], [U]))
    floor, eps = (1e-13 if prec == "FP64" else 1e-6), EPS[prec]
    th = sites[1].astype(np.complex128).reshape(chiL, -1)
    for j in range(1, k):
        th = (th.reshape(-1, chis[1 + j]) @ sites[1 + j].astype(np.complex128).reshape(chis[1 + j], -1))
    th = np.einsum("st,atb->asb", U, th.reshape(chiL, d, chiR))
    spectra, fw, want = _splits(th, lams[1], k, chi_max, floor)
    tol = 8 * eps * k * np.sqrt(max(chiL * d, 2 * chiR))
    dims = [int(x) for x in mps.bond_dims()]
    have = lams[1][:, None] * mps.site(1).astype(np.complex128).reshape(chiL, -1)
    for j in range(1, k):
        r = len(spectra[j])
        assert dims[1 + j] == r, (j, dims, r)
        np.testing.assert_allclose(mps.lam(1 + j), spectra[j], rtol=0, atol=tol)
        s = mps.site(1 + j).astype(np.complex128).reshape(r, -1)
        assert np.max(np.abs(s @ s.conj().T - np.eye(r))) <= tol
        have = have.reshape(-1, r) @ s
    assert abs(f - fw) <= tol
    have = have.reshape(chiL, -1)
    assert np.linalg.norm(have - want) <= tol * np.linalg.norm(want)


# (chi_L, chi_R, k): the splits are 2^j chi_L x at most 16, on both sides of that limit
SHAPES = [(1, 1, 2), (1, 8, 2), (2, 8, 2), (8, 8, 2), (8, 9, 2), (9, 1, 2), (3, 5, 3), (1, 1, 4), (2, 2, 3), (8, 1, 3),
          (1, 7, 5), (1, 1, 6), (33, 8, 2), (257, 8, 2), (350, 8, 2), (500, 8, 2)]


@pytest.mark.parametrize("prec", ["FP32", "FP64"])
@pytest.mark.parametrize("chiL,chiR,k", SHAPES)
def test_small_split_shapes(chiL, chiR, k, prec):
    _check(lib(), chiL, chiR, k, prec)


@pytest.mark.parametrize("prec", ["FP32", "FP64"])
@pytest.mark.parametrize("chiL,chiR,k,cap", [(8, 8, 2, 8), (5, 7, 3, 8), (1, 4, 5, 8), (3, 3, 4, 5)])
def test_small_split_truncates(chiL, chiR, k, cap, prec):
    """The inner bonds start narrow and the cut to chi_max bounds every later split's width."""
    P = lib()
    rng = np.random.default_rng(chiL + chiR + k)
    dtype = np.complex64 if prec == "FP32" else np.complex128
    chis = [1, chiL] + [2] * (k - 1) + [chiR, 1]
    sites = []
    for a, b in zip(chis[:-1], chis[1:]):
        g = rng.standard_normal((a, 2 * b)) + 1j * rng.standard_normal((a, 2 * b))
        sites.append((g / np.linalg.norm(g)).reshape(a, 2, b).astype(dtype))
    lams = [np.full(c, c ** -0.5) for c in chis]
    d = 2 ** k
    U = np.linalg.qr(rng.standard_normal((d, d)) + 1j * rng.standard_normal((d, d)))[0]
    mps = P.MPS(P.make_config(k + 2, cap, 0.0, 2 * k + 16, 0, k, getattr(P, prec)))
    mps.load(np.array(chis, dtype=np.int32), sites, lams)
    f = np.prod(mps.step([P.Cluster(1, k, 0, 0)], [U]))
    th = sites[1].astype(np.complex128).reshape(chiL, -1)
    for j in range(1, k):
        th = th.reshape(-1, 2) @ sites[1 + j].astype(np.complex128).reshape(2, -1)
    spectra, fw, _ = _splits(np.einsum("st,atb->asb", U, th.reshape(chiL, d, chiR)), lams[1], k, cap,
                             1e-13 if prec == "FP64" else 1e-6)
    tol = 8 * EPS[prec] * k * np.sqrt(max(chiL * d, 2 * chiR))
    dims = [int(x) for x in mps.bond_dims()]
    assert dims[2:1 + k] == [len(spectra[j]) for j in range(1, k)]
    assert max(dims) <= cap
    assert abs(f - fw) <= tol


@pytest.mark.parametrize("prec", ["FP32", "FP64"])
@pytest.mark.parametrize("chiL,chiR,k,rank", [(8, 8, 2, 1), (8, 8, 2, 3), (5, 5, 3, 2), (40, 8, 2, 5)])
def test_small_split_rank_deficient(chiL, chiR, k, rank, prec):
    _check(lib(), chiL, chiR, k, prec, inner=rank)
