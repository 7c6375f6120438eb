"""GPU: amplitudes of one stored state read by several threads at once (the
call takes a const state and releases the interpreter lock) are the ones that
one thread reads.  Short and wide bonds, so that calls with a lone CTA per half
and with many CTAs meet, and scratch grows while others read.

The kernel sums in a fixed order: the values are equal, bit for bit."""
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import pytest

from gpu_helpers import lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["FP32", "FP64"])
@pytest.mark.parametrize("chi", [8, 96])
def test_threads_read_the_amplitudes_one_thread_reads(chi, prec):
    P = lib()
    n, threads, each = 24, 4, 16
    rng = np.random.default_rng(chi)
    chis = np.array([min(chi, 2 ** min(b, n - b)) for b in range(n + 1)], dtype=np.int32)
    dt = np.complex64 if prec == "FP32" else np.complex128
    sites = []
    for q in range(n):
        g = rng.standard_normal((chis[q], 2, chis[q + 1])) + 1j * rng.standard_normal((chis[q], 2, chis[q + 1]))
        sites.append((g / np.linalg.norm(g, 2, axis=(0, 2)).max()).astype(dt))
    cfg = P.make_config(n, chi, 0.0, 4 + 2 * int(np.ceil(np.log2(chi))), 0, 2, getattr(P, prec))

    def state():
        mps = P.MPS(cfg)
        mps.load(chis, sites, [np.ones(c) / np.sqrt(c) for c in chis])
        return mps

    bits = rng.integers(0, 2, (threads, each, n)).astype(np.uint8)
    alone = state()
    want = np.array([[alone.amplitude(b) for b in row] for row in bits])
    shared = state()                      # no scratch yet: the first calls make it
    with ThreadPoolExecutor(threads) as pool:
        got = list(pool.map(lambda row: [shared.amplitude(b) for b in row], bits))
    np.testing.assert_array_equal(np.array(got), want)
