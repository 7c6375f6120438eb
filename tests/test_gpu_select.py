"""GPU: the truncation's sort, suffix sums and cut on spectra that are known
beforehand -- theta = Q1 diag(d) Q2 with a flat left spectrum -- at the edges
of a warp, of the block and of the positions per thread, with ties and with
numerical zeros behind the rank, with and without a cutoff.

Weights differ by at least a factor of two between groups and every cut lies a
factor of 1.3 from the nearest tail sum, so the rank is exact; the spectrum has
the split's backward error, 8 eps sqrt(n)."""
import numpy as np
import pytest

from gpu_helpers import lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["FP32", "FP64"])
@pytest.mark.parametrize("r", [1, 17, 31, 32, 33, 64, 65, 513, 1024])
def test_known_spectra(r, prec):
    P = lib()
    if r > 600 and prec == "FP64":
        pytest.skip("the same kernel as in FP32")
    rng = np.random.default_rng(r)
    a = max(r, 9)                                      # 2a x 2a matrices of rank r
    eps = 2.0 ** -23 if prec == "FP32" else 2.0 ** -52

    def iso(rows):
        return np.linalg.qr(rng.standard_normal((rows, r)) + 1j * rng.standard_normal((rows, r)))[0]

    # groups of equal weights, each 1/8 of the group before
    group = max(1, (r + 4) // 5)
    p = 8.0 ** -(np.arange(r) // group)
    p /= p.sum()
    q1, q2 = iso(2 * a), iso(2 * a)
    dtype = np.complex64 if prec == "FP32" else np.complex128
    chis = [1, a, r, a, 1]
    sites = [np.ones((1, 2, a)) / np.sqrt(2 * a), (q1 * np.sqrt(p)).reshape(a, 2, r), q2.conj().T.reshape(r, 2, a),
             np.ones((a, 2, 1)) / np.sqrt(2 * a)]
    sites = [s.astype(dtype) for s in sites]
    lams = [np.full(c, c ** -0.5) for c in chis]
    tails = np.append(np.cumsum(p[::-1])[::-1], 0.0)   # weight from position i on
    for cutoff in (0.0, 1.3 * tails[min(r, 3 * group)], 0.7 * tails[min(2 * group, r - 1)]):
        lg = int(np.ceil(np.log2(2 * a)))
        mps = P.MPS(P.make_config(4, 2 * a, min(float(cutoff), 0.9), 2 + 2 * lg, 0, 2, getattr(P, prec)))
        mps.load(np.array(chis, dtype=np.int32), sites, lams)
        f = mps.step([P.Cluster(1, 2, 0, 0)], [np.eye(4, dtype=np.complex128)])[0]
        want = r
        if cutoff > 0:
            want = max(1, int(np.argmax(tails <= min(float(cutoff), 0.9))))
        tol = 8 * eps * np.sqrt(2 * a)
        got = int(mps.bond_dims()[2])
        if cutoff > 0 and want % group and want < r:   # a cut inside a group of equal weights: any of them
            assert abs(got - want) <= 1
            continue
        assert got == want, (r, cutoff, got, want)
        assert abs(f - p[:want].sum()) <= tol
        np.testing.assert_allclose(mps.lam(2), np.sqrt(p[:want] / p[:want].sum()), rtol=0, atol=tol)
