"""GPU: splits with very many rows -- wide clusters of many qubits, beyond what
the direct solver's per-row scratch takes (2^18 to 2^19 rows of an 8-qubit
right part) -- are accepted and exact, and a step after them works as before.

The state has inner bonds of 4, so every bond's spectrum follows from 4 x 4
products of the left and right environments, in FP64 on the host.

Tolerances: a kept direction that is off by a relative d changes weights in
second order, and FP32 sums over 2^19 rows are good to about 2^-23 sqrt(2^19) =
9e-5: 1e-7 for fidelities and 2e-6 for the spectra of the FP32 mode (as in the
other wide-cluster tests), 1e-12 and 1e-11 in FP64."""
import numpy as np
import pytest

from gpu_helpers import lib

pytestmark = pytest.mark.gpu


def _spectra(lam, sites, q0, k):
    """Schmidt spectra of the bonds inside a cluster, from environments."""
    left = np.diag(lam.astype(np.complex128) ** 2)
    lefts = []
    for q in range(q0, q0 + k - 1):
        s = sites[q].astype(np.complex128)
        left = np.einsum("ab,asc,bsd->cd", left, s.conj(), s, optimize=True)
        lefts.append(left)
    right = np.eye(sites[q0 + k - 1].shape[2], dtype=np.complex128)
    out = []
    for q in range(q0 + k - 1, q0, -1):
        s = sites[q].astype(np.complex128)
        right = np.einsum("asc,cd,bsd->ab", s, right, s.conj(), optimize=True)
        w = np.sort(np.linalg.eigvals(lefts[q - 1 - q0] @ right).real)[::-1]
        out.append(np.sqrt(w / w.sum()))
    return out[::-1]


def _overlap(lam, a, b):
    """<a|b> of two clusters' theta."""
    t = np.diag(lam.astype(np.complex128) ** 2)
    for x, y in zip(a, b):
        t = np.einsum("ab,asc,bsd->cd", t, x.astype(np.complex128).conj(), y.astype(np.complex128), optimize=True)
    return np.trace(t)


# (precision, chi_L, k, chi_R): first split chi_L 2^(k - 1) x 2 chi_R
CASES = [("FP64", 2048, 9, 8), ("FP64", 1024, 9, 33), ("FP32", 2048, 9, 129)]


@pytest.mark.parametrize("prec,chi_l,k,chi_r", CASES)
def test_split_with_very_many_rows(prec, chi_l, k, chi_r):
    P = lib()
    rng = np.random.default_rng(chi_r)
    inner = 4
    chis = np.array([1, chi_l] + [inner] * (k - 1) + [chi_r, 1], dtype=np.int32)
    dt = np.complex64 if prec == "FP32" else np.complex128
    sites = []
    for a, b in zip(chis, chis[1:]):
        g = rng.standard_normal((a, 2, b)) + 1j * rng.standard_normal((a, 2, b))
        sites.append((g / np.linalg.norm(g)).astype(dt))
    lams = [np.ones(c) / np.sqrt(c) for c in chis]
    n = len(sites)
    cutoff = 1e-8 if prec == "FP32" else 1e-13
    cfg = P.make_config(n, chi_l, cutoff, k + 2 * 11, 0, k, getattr(P, prec))
    mps = P.MPS(cfg)
    mps.load(chis, sites, lams)
    f = mps.step([P.Cluster(1, k, 0, 0)], [np.eye(1 << k, dtype=np.complex128)])
    tol_f, tol_lam = (1e-7, 2e-6) if prec == "FP32" else (1e-12, 1e-11)
    assert np.all(np.abs(f - 1) <= tol_f), f
    want = _spectra(lams[1], sites, 1, k)
    for j in range(1, k):
        got = mps.lam(1 + j)
        assert len(got) == inner
        np.testing.assert_allclose(got, want[j - 1], rtol=0, atol=tol_lam)
    new = [mps.site(q) for q in range(1, 1 + k)]
    old = sites[1:1 + k]
    ov = abs(_overlap(lams[1], old, new))
    norm = np.sqrt(abs(_overlap(lams[1], old, old)) * abs(_overlap(lams[1], new, new)))
    assert abs(ov / norm - 1) <= tol_f
    # the handle is good for an ordinary step afterwards
    f = mps.step([P.Cluster(2, 2, 0, 0)], [np.eye(4, dtype=np.complex128)])
    assert abs(f[0] - 1) <= tol_f
