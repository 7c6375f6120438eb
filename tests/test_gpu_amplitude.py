"""GPU: amplitudes of stored states against the same chain in numpy, where the
kernel's split of the work changes: one site, a lone CTA per half, several
CTAs, bonds that leave CTAs without a slice (a narrow waist after wide bonds),
more values per thread than are read ahead, both precisions.

Tolerance: both sides multiply the same stored values and accumulate in FP64
over n <= 60 sites, so they agree to about n chi eps64 of the vectors' norms;
1e-11 of the product of the sites' norms bounds it."""
import numpy as np
import pytest

from gpu_helpers import lib

pytestmark = pytest.mark.gpu

BONDS = {
    "one site": [1, 1],
    "two sites": [1, 2, 1],
    "lone CTA": [1] + [7, 20, 31, 5, 32, 17] * 4 + [1],
    "several CTAs": [1] + [40, 64, 37, 64] * 6 + [1],
    "waist": [1] + [120, 120, 2, 1, 3, 120, 128] * 5 + [1],
    "wide": [1, 300, 512, 511, 512, 1],
}


@pytest.mark.parametrize("prec", ["FP32", "FP64"])
@pytest.mark.parametrize("bonds", sorted(BONDS))
def test_amplitude_matches_numpy(bonds, prec):
    P = lib()
    chis = np.array(BONDS[bonds], dtype=np.int32)
    n = len(chis) - 1
    rng = np.random.default_rng(n)
    dt = np.complex64 if prec == "FP32" else np.complex128
    sites = []
    for q in range(n):
        g = rng.standard_normal((chis[q], 2, chis[q + 1])) + 1j * rng.standard_normal((chis[q], 2, chis[q + 1]))
        sites.append((g / np.linalg.norm(g, 2, axis=(0, 2)).max()).astype(dt))
    lams = [np.ones(c) / np.sqrt(c) for c in chis]
    top = int(chis.max())
    cfg = P.make_config(n, top, 0.0, 4 + 2 * int(np.ceil(np.log2(max(top, 2)))), 0, 2, getattr(P, prec))
    mps = P.MPS(cfg)
    mps.load(chis, sites, lams)
    for _ in range(3):
        bits = rng.integers(0, 2, n).astype(np.uint8)
        v, scale = np.ones(1, dtype=np.complex128), 1.0
        for s, b in zip(sites, bits):
            m = s[:, b, :].astype(np.complex128)
            v = v @ m
            scale *= np.linalg.norm(m)
        assert abs(mps.amplitude(bits) - v[0]) <= 1e-11 * scale
    with pytest.raises(P.CtebdError):
        mps.amplitude(np.full(n, 2, np.uint8))
