"""GPU: tall splits in a level with many of them take the Gram matrix and
Jacobi, one of them alone the direct solver; both give the same state.

Sixteen clusters of seven qubits, 64 wide on both sides (first split 4096 x
128), in one step and one cluster at a time.  The inner bonds are 64 wide as
well, so nothing but rounding is dropped and theta must come back.

Tolerances: the Gram matrix resolves weights to eps |M|^2 (FP32 after the
refinement pass: relative to each weight), so with weights of at least 1e-4 of
the largest theta is good to 1e2 eps n: 5e-5 in FP32 (as for the other Jacobi
tests) and 1e-11 in FP64; weights are of second order in that."""
import numpy as np
import pytest

from gpu_helpers import lib

pytestmark = pytest.mark.gpu

CHI, K, COUNT = 64, 7, 16


def _cluster_theta(lam, sites):
    t = lam[:, None] * sites[0].reshape(sites[0].shape[0], -1).astype(np.complex128)
    for s in sites[1:]:
        t = t.reshape(-1, s.shape[0]) @ s.reshape(s.shape[0], -1).astype(np.complex128)
    return t.reshape(-1)


@pytest.mark.parametrize("prec", ["FP32", "FP64"])
def test_tall_splits_together_and_alone(prec):
    P = lib()
    rng = np.random.default_rng(17)
    dt = np.complex64 if prec == "FP32" else np.complex128
    chis = np.array([1] + [CHI] * (COUNT * K + 1) + [1], dtype=np.int32)
    sites = []
    for a, b in zip(chis, chis[1:]):
        g = rng.standard_normal((2 * b, a)) + 1j * rng.standard_normal((2 * b, a))
        g = np.linalg.qr(g)[0] if a <= 2 * b else g / np.linalg.norm(g)
        sites.append(np.ascontiguousarray(g.conj().T).reshape(a, 2, b).astype(dt))
    lams = []
    for c in chis:
        w = np.sort(rng.uniform(0.05, 1.0, c))[::-1]
        lams.append(np.sqrt(w / w.sum()))
    cfg = P.make_config(len(sites), CHI, 1e-10 if prec == "FP32" else 1e-20, K + 12, 0, K, getattr(P, prec))
    eye = np.eye(1 << K, dtype=np.complex128)
    q0s = [1 + i * K for i in range(COUNT)]
    clusters = [P.Cluster(q, K, 0, 0) for q in q0s]
    together = P.MPS(cfg)
    together.load(chis, sites, lams)
    f = together.step(clusters, [eye] * COUNT)
    log = together.split_log()
    first = log[log[:, 3] == CHI << (K - 1)]
    assert len(first) == COUNT and np.all(first[:, 4] == 2 * CHI)
    assert np.all(first[:, 12] > 0)              # Jacobi sweeps
    assert np.all(log[log[:, 3] < 8 * log[:, 4], 12] == 0)
    one = P.MPS(cfg)
    one.load(chis, sites, lams)
    for i in (0, COUNT - 1):
        one.step([clusters[i]], [eye])
        assert np.all(one.split_log()[:, 12] == 0)   # the direct solver
    tol = 5e-5 if prec == "FP32" else 1e-11
    assert np.all(np.abs(f - 1) <= tol), f
    for i in (0, COUNT - 1):
        q = q0s[i]
        want = _cluster_theta(lams[q], sites[q:q + K])
        s = np.linalg.svd(want.reshape(-1, 2 * CHI), compute_uv=False)[:CHI]
        for m in (together, one):
            assert list(m.bond_dims()[q:q + K + 1]) == [CHI] * (K + 1)
            got = _cluster_theta(lams[q], [m.site(x) for x in range(q, q + K)])
            assert np.linalg.norm(got - want) <= tol * np.linalg.norm(want)
            np.testing.assert_allclose(m.lam(q + K - 1), s / np.linalg.norm(s), rtol=0, atol=tol)
