"""GPU: a call that is refused half-way leaves work behind on the handle's
stream.  The calls after it wait for that before they use the staging memory
again, and give what a fresh handle gives.

The refused call is a step whose second cluster has ten qubits (its unitary
exceeds the staging block), after the first one's products were queued.  The
same kernels run on the same inputs: values are equal bit for bit."""
import numpy as np
import pytest

from gpu_helpers import lib, random_unitary

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("after", ["amplitude", "step", "load_device"])
def test_calls_after_a_refused_step(after):
    P = lib()
    import torch
    rng = np.random.default_rng(5)
    chi, tail = 384, 10
    chis = np.array([1, chi, chi, chi, chi] + [1] * (tail + 1), dtype=np.int32)
    n = len(chis) - 1
    sites = []
    for a, b in zip(chis, chis[1:]):
        g = rng.standard_normal((a, 2, b)) + 1j * rng.standard_normal((a, 2, b))
        sites.append((g / np.linalg.norm(g, 2, axis=(0, 2)).max()).astype(np.complex64))
    lams = [np.ones(c) / np.sqrt(c) for c in chis]
    cfg = P.make_config(n, chi, 1e-8, 2 + 2 * 9, 0, tail, P.FP32)
    pair = P.Cluster(2, 2, 0, 0)
    U = random_unitary(4, rng)
    bits = rng.integers(0, 2, (4, n)).astype(np.uint8)
    dev = [torch.from_numpy(x).cuda() for x in sites], [torch.from_numpy(x).cuda() for x in lams]
    torch.cuda.synchronize()

    def use(mps):
        if after == "load_device":
            mps.load_device(chis, [x.data_ptr() for x in dev[0]], [x.data_ptr() for x in dev[1]])
        if after == "step":
            mps.step([pair], [U])
        return [mps.amplitude(b) for b in bits], mps.lam(3)

    fresh = P.MPS(cfg)
    fresh.load(chis, sites, lams)
    want, lam = use(fresh)
    mps = P.MPS(cfg)
    mps.load(chis, sites, lams)
    with pytest.raises(P.CtebdError, match="staging"):
        mps.step([P.Cluster(1, 2, 0, 0), P.Cluster(n - tail, tail, 0, 0)], [U, np.eye(1 << tail, dtype=np.complex128)])
    got, lam2 = use(mps)
    np.testing.assert_array_equal(got, want)
    np.testing.assert_array_equal(lam2, lam)
