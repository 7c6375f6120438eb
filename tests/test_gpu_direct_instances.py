"""GPU: instances of the direct split's kernels that ordinary sizes do not reach
-- rows that do not fit the chip's shared memory (wide and narrow matrices),
more than 2048 (FP32) or 1024 (FP64) columns, the widest back-transformations,
and the smallest problems behind a wide first split -- against numpy's SVD.

Which kernels ran is read from the launch counts.  On 152 SMs the plan keeps
these rows in global memory: FP64 2560 x 1280, 1030 x 2050, 8192 x 130, 32768 x
34; FP32 2200 x 2050, 4096 x 1026, 16384 x 130, 65536 x 34.

Tolerances: as for the direct split of ordinary sizes, 8 eps sqrt(rows or
columns), of which f is good to the square."""
import ctypes as C

import numpy as np
import pytest

from gpu_helpers import lib, random_unitary
from test_gpu_direct_split import EPS, _state, _site

pytestmark = pytest.mark.gpu


def _launches(P, mps):
    rows, n = np.zeros(5 * 32), C.c_int(0)
    P._check(P.lib.ctebd_profile_read(mps._h, rows.ctypes.data_as(C.POINTER(C.c_double)), 32, C.byref(n)), "profile")
    out = {}
    for k in range(n.value):
        buf = C.create_string_buffer(64)
        P.lib.ctebd_kernel_name(k, buf, 64)
        out[buf.value.decode()] = int(rows[5 * k])
    return out


def _theta(lam, sites):
    t = lam[:, None] * sites[0].astype(np.complex128).reshape(len(lam), -1)
    for s in sites[1:]:
        t = t.reshape(-1, s.shape[0]) @ s.astype(np.complex128).reshape(s.shape[0], -1)
    return t


def _run(prec, chis, sites, lams, q0, k, U, chi_max, cutoff):
    """One cluster; checks that the direct solver did every split, and the first split against numpy."""
    P = lib()
    top = max(chi_max, int(max(chis)))
    cfg = P.make_config(len(sites), top, cutoff, k + 2 * int(np.ceil(np.log2(top))) + 2, 0, k, getattr(P, prec))
    mps = P.MPS(cfg)
    mps.load(chis, sites, lams)
    P._check(P.lib.ctebd_profile(mps._h, 0), "profile")
    f = mps.step([P.Cluster(q0, k, 0, 0)], [U])
    n = _launches(P, mps)
    assert n["bidiag"] == k - 1 and n["small_chain"] == 0 and n["eig_inner"] == 0, n
    a, c = int(chis[q0]), int(chis[q0 + k])
    th = _theta(lams[q0], sites[q0:q0 + k]).reshape(a, 1 << k, c)
    th = np.matmul(U, th).reshape(-1, 2 * c)
    u, s, vh = np.linalg.svd(th, full_matrices=False)
    p = s * s
    tol = 8 * EPS[prec] * np.sqrt(max(th.shape))
    r = int(mps.bond_dims()[q0 + k - 1])
    np.testing.assert_allclose(mps.lam(q0 + k - 1), s[:r] / np.sqrt(p[:r].sum()), rtol=0, atol=tol)
    assert abs(f[0] - p[:r].sum() / p.sum()) <= max(tol, 4 * EPS[prec])
    right = mps.site(q0 + k - 1).astype(np.complex128).reshape(r, -1)
    assert np.max(np.abs(right @ right.conj().T - np.eye(r))) <= tol
    if k == 2:
        left = mps.site(q0).astype(np.complex128)
        want = (u[:, :r] * s[:r]) @ vh[:r] / np.sqrt(p[:r].sum())
        have = (lams[q0][:, None] * left.reshape(a, -1)).reshape(2 * a, r) @ right
        assert np.linalg.norm(have - want) <= tol * np.linalg.norm(want)
    return mps, r


# precision, chi_L, middle bond, chi_R: the split is 2 chi_L x 2 chi_R
PAIRS = [("FP64", 1280, 700, 640),    # 8 columns a thread, rows in global memory
         ("FP64", 100, 120, 1025),    # 16 columns a thread
         ("FP64", 515, 520, 1025),    # 16, rows in global memory
         ("FP32", 100, 120, 1025),    # 8 columns a thread
         ("FP32", 1100, 1400, 1025),  # 8, rows in global memory
         ("FP32", 2048, 700, 513),    # 4, rows in global memory
         ("FP32", 32, 40, 2048),      # 4096 columns: 4 columns of V a CTA
         ("FP64", 32, 40, 2048)]      # 2 columns of V a CTA


@pytest.mark.parametrize("prec,a,b,c", PAIRS)
def test_wide_and_nonresident_pairs(prec, a, b, c):
    rng = np.random.default_rng(a + c)
    chis, sites, lams = _state(rng, [(a, b, c)], np.complex64 if prec == "FP32" else np.complex128)
    _, r = _run(prec, chis, sites, lams, 1, 2, random_unitary(4, rng), min(2 * a, 2 * c, 2048), 0.0)
    assert r == min(2 * a, 2 * c, 2048)


@pytest.mark.parametrize("prec,a,k,c", [("FP32", 1024, 5, 65), ("FP32", 1024, 7, 17), ("FP64", 512, 5, 65),
                                        ("FP64", 1024, 6, 17)])
def test_narrow_rows_in_global_memory(prec, a, k, c):
    """Several rows of threads per CTA and rows in global memory: tall, narrow first splits."""
    rng = np.random.default_rng(a + c)
    dt = np.complex64 if prec == "FP32" else np.complex128
    chis = np.array([1, a] + [c] * k + [1], dtype=np.int32)
    sites = [_site(rng, x, y).astype(dt) for x, y in zip(chis, chis[1:])]
    lams = []
    for x in chis:
        w = np.sort(rng.exponential(1.0, x))[::-1]
        lams.append(np.sqrt(w / w.sum()))
    _run(prec, chis, sites, lams, 1, k, random_unitary(1 << k, rng), c, 0.0)


@pytest.mark.parametrize("prec", ["FP32", "FP64"])
@pytest.mark.parametrize("inner", [1, 2, 3, 4, 5, 8])
def test_smallest_problems_behind_a_wide_split(inner, prec):
    """Second splits of 2 to 16 columns by the direct solver: no merge, one merge."""
    rng = np.random.default_rng(inner)
    dt = np.complex64 if prec == "FP32" else np.complex128
    chis = np.array([1, 40, inner, inner, 20, 1], dtype=np.int32)
    sites = [_site(rng, x, y).astype(dt) for x, y in zip(chis, chis[1:])]
    lams = []
    for x in chis:
        w = np.sort(rng.uniform(0.2, 1.0, x))[::-1]
        lams.append(np.sqrt(w / w.sum()))
    mps, r = _run(prec, chis, sites, lams, 1, 3, np.eye(8, dtype=np.complex128), 40, 1e-9 if prec == "FP32" else 1e-20)
    assert r == inner and mps.bond_dims()[2] == inner
    want = _theta(lams[1], sites[1:4]).reshape(-1)
    have = _theta(lams[1], [mps.site(q) for q in (1, 2, 3)]).reshape(-1)
    assert np.linalg.norm(have / np.linalg.norm(have) - want / np.linalg.norm(want)) <= 8 * EPS[prec] * np.sqrt(80)
