"""GPU: states in and out of the handle -- exact round trips through the batched
device copy (aligned to 16 bytes and to 8 only, page-locked host sources among
device ones), reads on both sides of the size where the host widens FP32
itself, and unitaries larger than the first staging block."""
import numpy as np
import pytest
import torch

from gpu_helpers import lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["FP32", "FP64"])
@pytest.mark.parametrize("chis", [[1, 1], [1, 2, 3, 1], [1, 90, 91, 91, 1], [1, 7, 300, 301, 1]])
@pytest.mark.parametrize("shift", [0, 8])
def test_load_device_round_trip(chis, shift, prec):
    P = lib()
    rng = np.random.default_rng(sum(chis))
    dtype = torch.complex64 if prec == "FP32" else torch.complex128
    keep, sp, lp, sites, lams = [], [], [], [], []

    def put(a, pinned):
        raw = np.frombuffer(np.ascontiguousarray(a).tobytes(), dtype=np.uint8)
        t = torch.zeros(len(raw) + shift, dtype=torch.uint8, pin_memory=pinned, device="cpu" if pinned else "cuda")
        t[shift:] = torch.from_numpy(raw.copy())
        keep.append(t)
        return t.data_ptr() + shift

    for q, (a, b) in enumerate(zip(chis[:-1], chis[1:])):
        s = torch.from_numpy(rng.standard_normal((a, 2, b)) + 1j * rng.standard_normal((a, 2, b))).to(dtype).numpy()
        sites.append(s)
        sp.append(put(s, q % 3 == 2))
    for b, c in enumerate(chis):
        lams.append(rng.random(c))
        lp.append(put(lams[-1], b % 2 == 1))
    torch.cuda.synchronize()
    n = len(chis) - 1
    mps = P.MPS(P.make_config(n, 512, 0.0, 2 + 2 * 9, 0, 2, getattr(P, prec)))
    mps.load_device(np.array(chis, dtype=np.int32), sp, lp)
    for q in range(n):
        np.testing.assert_array_equal(mps.site(q), sites[q].astype(np.complex128))
    for b in range(n + 1):
        np.testing.assert_array_equal(mps.lam(b), lams[b])


@pytest.mark.parametrize("prec", ["FP32", "FP64"])
@pytest.mark.parametrize("ks", [(9, 9), (8, 4, 8, 2, 9), (2,) * 300])
def test_unitaries_larger_than_first_staging_block(ks, prec):
    """X on the first qubit of every cluster, by whole-cluster unitaries: exact in both precisions."""
    P = lib()
    n = sum(ks)
    mps = P.MPS(P.make_config(n, 4, 0.0, 2 * max(ks) + 4, 0, max(ks), getattr(P, prec)))
    cl, Us, q = [], [], 0
    for k in ks:
        D = 1 << k
        cl.append(P.Cluster(q, k, 0, 0))
        Us.append(np.roll(np.eye(D, dtype=np.complex128), D // 2, axis=0))
        q += k
    f = mps.step(cl, Us)
    np.testing.assert_allclose(f, 1.0, rtol=0, atol=0)
    bits = np.zeros(n, dtype=np.uint8)
    for c in cl:
        bits[c.q0] = 1
    assert abs(abs(mps.amplitude(bits)) - 1) <= n * 2.0 ** -23
    assert list(mps.bond_dims()) == [1] * (n + 1)
