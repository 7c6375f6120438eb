"""GPU: the Gram matrix and Jacobi path of full splits, where it is the one that
runs -- tall splits of wide clusters, the forced tensor-core policy, a sweep cap
below the direct solver's.  Every test asserts from the split log that Jacobi
sweeps were made.

- The sweep loop on the device (CUDA graph with a WHILE node) and from the host
  run the same kernels in the same order: equal ranks and sweep counts, and
  fidelities equal to rounding; bit for bit in the batch that takes the compact
  tail (more than eight problems, 32 blocks wide).
- Accuracy against numpy's SVD, on the CUDA cores and on the tensor cores:
  in FP32 1e-5 of the kept weight and 1e-3 relative and 2e-6 absolute of the
  spectrum, as in the tests of the tensor-core round update, 1e-11 in FP64."""
import numpy as np
import pytest

from gpu_helpers import lib, random_unitary

pytestmark = pytest.mark.gpu


class _State:
    """Clusters side by side, sites random right isometries, made on the device."""

    def __init__(self, P, prec, chi, k, count, chi_max, cutoff, seed):
        import torch
        self.P, self.k = P, k
        dt = torch.complex64 if prec == "FP32" else torch.complex128
        gen = torch.Generator(device="cuda")
        gen.manual_seed(seed)
        rng = np.random.default_rng(seed)
        ramp = [1]
        while 2 * ramp[-1] < chi:
            ramp.append(2 * ramp[-1])
        self.chis = np.array(ramp + [chi] * (count * k + 1) + ramp[::-1], dtype=np.int32)
        c = self.chis.tolist()
        self.sites = [torch.linalg.qr(torch.randn(2 * b, a, dtype=dt, device="cuda", generator=gen))[0]
                      .conj().resolve_conj().t().contiguous() for a, b in zip(c, c[1:])]
        self.lams = []
        for x in c:
            w = np.sort(rng.exponential(1.0, x))[::-1]
            self.lams.append(torch.from_numpy(np.sqrt(w / w.sum()).copy()).cuda())
        self.q0s = [len(ramp) + i * k for i in range(count)]
        self.Us = [random_unitary(1 << k, rng) for _ in range(count)]
        lg = int(np.ceil(np.log2(max(chi_max, chi))))
        self.cfg = P.make_config(len(c) - 1, max(chi_max, chi), cutoff, k + 2 * lg, 0, k, getattr(P, prec))
        torch.cuda.synchronize()

    def step(self, graphs=None, mode=1, cap=60):
        P = self.P
        old = P.max_sweeps()
        try:
            if graphs is not None:
                P.set_sweep_graphs(2 if graphs else 0)
            P.set_tensor_cores(mode)
            P.set_max_sweeps(cap)
            mps = P.MPS(self.cfg)
            mps.load_device(self.chis, [x.data_ptr() for x in self.sites], [x.data_ptr() for x in self.lams])
            f = mps.step([P.Cluster(q, self.k, 0, 0) for q in self.q0s], self.Us)
            return mps, f, mps.split_log()
        finally:
            P.set_sweep_graphs(1)
            P.set_tensor_cores(1)
            P.set_max_sweeps(old)

    def theta(self, i):
        q, k = self.q0s[i], self.k
        t = self.sites[q].cpu().numpy().astype(np.complex128)
        a = t.shape[0]
        for j in range(1, k):
            s = self.sites[q + j].cpu().numpy().astype(np.complex128)
            t = t.reshape(-1, s.shape[0]) @ s
        t = t.reshape(a, 1 << k, -1)
        return self.lams[q].cpu().numpy()[:, None, None] * np.einsum("st,atb->asb", self.Us[i], t)


# precision, chi, k, clusters, tensor-core policy, sweep cap; first split chi 2^(k - 1) x 2 chi
LOOPS = [("FP32", 64, 7, 16, 1, 60), ("FP64", 64, 7, 16, 1, 60), ("FP32", 256, 9, 1, 1, 60), ("FP32", 128, 2, 2, 2, 60),
         ("FP64", 100, 2, 3, 2, 60), ("FP32", 48, 2, 3, 0, 11)]


@pytest.mark.parametrize("prec,chi,k,count,mode,cap", LOOPS)
def test_sweep_loop_on_device_and_host(prec, chi, k, count, mode, cap):
    s = _State(lib(), prec, chi, k, count, chi, 1e-8, seed=chi + k)
    (m_g, f_g, log_g), (m_h, f_h, log_h) = (s.step(g, mode, cap) for g in (True, False))
    first = log_g[:, 3] == chi << (k - 1)
    assert first.sum() == count and np.all(log_g[first, 12] > 0)
    assert list(m_g.bond_dims()) == list(m_h.bond_dims())
    np.testing.assert_array_equal(log_g[:, [5, 12, 13]], log_h[:, [5, 12, 13]])   # ranks, sweeps of both passes
    np.testing.assert_allclose(f_g, f_h, rtol=1e-9)


def test_compact_tail_on_device_and_host():
    s = _State(lib(), "FP32", 512, 6, 9, 512, 1e-8, seed=9)
    (m_g, f_g, log_g), (m_h, f_h, log_h) = (s.step(g) for g in (True, False))
    first = (log_g[:, 3] == 512 << 5) & (log_g[:, 4] == 1024)
    assert first.sum() == 9 and np.all(log_g[first, 12] > 0)
    np.testing.assert_array_equal(log_g[:, [5, 12, 13]], log_h[:, [5, 12, 13]])
    np.testing.assert_array_equal(f_g, f_h)


# the CUDA cores (policies 0 and 1, and a cap below the direct solver's) and the tensor cores (policy 2)
ACCURACY = [("FP32", 64, 7, 16, 0, 60), ("FP32", 64, 7, 16, 2, 60), ("FP64", 64, 7, 16, 1, 60), ("FP32", 64, 2, 2, 0, 11),
            ("FP64", 32, 2, 2, 1, 11), ("FP64", 64, 2, 2, 2, 60)]


@pytest.mark.parametrize("prec,chi,k,count,mode,cap", ACCURACY)
def test_jacobi_split_matches_svd(prec, chi, k, count, mode, cap):
    s = _State(lib(), prec, chi, k, count, chi, 1e-8, seed=2 * chi + k)
    mps, f, log = s.step(None, mode, cap)
    for i in (0, count - 1):
        q = s.q0s[i]
        row = log[(log[:, 0] == q) & (log[:, 2] == q + k - 1)][0]
        assert row[12] > 0
        p = np.linalg.svd(s.theta(i).reshape(-1, 2 * chi), compute_uv=False) ** 2
        r = int(mps.bond_dims()[q + k - 1])
        assert r == min(chi, int(row[5]))
        assert abs(row[6] - p[:r].sum() / p.sum()) <= (1e-5 if prec == "FP32" else 1e-11)
        np.testing.assert_allclose(mps.lam(q + k - 1), np.sqrt(p[:r] / p[:r].sum()),
                                   rtol=1e-3 if prec == "FP32" else 0, atol=2e-6 if prec == "FP32" else 1e-11)


@pytest.mark.parametrize("chi_l,chi_r,chi_max", [(16, 16, 32), (32, 40, 24), (64, 48, 64)])
def test_noalloc_jacobi_branch_matches_svd(chi_l, chi_r, chi_max):
    """A sweep cap below the direct solver's: split2_noalloc takes its Gram and Jacobi branch."""
    import torch
    P = lib()
    rng = np.random.default_rng(chi_l)
    th = rng.standard_normal((chi_l, 4, chi_r)) + 1j * rng.standard_normal((chi_l, 4, chi_r))
    th = (th / np.linalg.norm(th)).astype(np.complex64)
    lam = np.sort(rng.uniform(0.2, 1.0, chi_l))[::-1]
    lam = lam / np.linalg.norm(lam)
    p = np.linalg.svd((lam[:, None, None] * th.astype(np.complex128)).reshape(2 * chi_l, 2 * chi_r), compute_uv=False) ** 2
    theta = torch.from_numpy(th).cuda()
    lam_d = torch.from_numpy(lam.copy()).cuda()
    left = torch.zeros(2 * chi_l * chi_max, dtype=torch.complex64, device="cuda")
    right = torch.zeros(chi_max * 2 * chi_r, dtype=torch.complex64, device="cuda")
    spec = torch.zeros(chi_max, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    old = P.max_sweeps()
    try:
        P.set_max_sweeps(11)
        r, f = P.split2_noalloc(theta.data_ptr(), lam_d.data_ptr(), chi_l, chi_r, chi_max, 1e-8,
                                left.data_ptr(), right.data_ptr(), spec.data_ptr())
    finally:
        P.set_max_sweeps(old)
    assert r == min(chi_max, len(p))
    assert abs(f - p[:r].sum() / p.sum()) <= 1e-5
    np.testing.assert_allclose(spec.cpu().numpy()[:r], np.sqrt(p[:r] / p[:r].sum()), rtol=1e-3, atol=2e-6)
    B = right.cpu().numpy()[: r * 2 * chi_r].reshape(r, -1).astype(np.complex128)
    assert np.max(np.abs(B @ B.conj().T - np.eye(r))) <= 5e-5
