"""GPU: the scalar routines of numeric.cuh and pair.cuh (square root and
reciprocal by Newton's iteration, in FP32, FP64 and pairs of FP32 numbers)
against extended precision, over the ranges that their comments state.

Bounds (derived there): half an ulp and a fiftieth of it, 1.02 x 2^-24 and
1.02 x 2^-53 relative, and 2^-44 for pairs.

Also here: a bounded wait of exchange.cuh on a slot that nothing fills ends, and
says which kernel waited."""
import os
import subprocess

import numpy as np
import pytest

import paper_2502_19289_gb300.build as B

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("probe") / "numeric_probe")
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "numeric_probe.cu")
    subprocess.run([B._nvcc()] + B.ARCH + ["-O3", "-std=c++17", "--expt-relaxed-constexpr", "-I", B.CSRC, src, "-o", out],
                   check=True, capture_output=True)
    return out


def _arguments(lo, hi, single):
    rng = np.random.default_rng(1)
    x = np.exp(rng.uniform(np.log(lo), np.log(hi), 200000))
    one = np.concatenate([1 + np.arange(-64, 65) * 2.0 ** -24, 1 + np.arange(-64, 65) * 2.0 ** -53,
                          2.0 ** np.arange(-60.0, 61.0)])
    x = np.concatenate([x, one, 2 * one, rng.uniform(1.0, 4.0, 200000)])
    return x.astype(np.float32).astype(np.float64) if single else x


CASES = {  # lowest and highest argument, arguments rounded to FP32, bound
    "sqrt32": (1e-36, 1e37, True, 1.02 * 2.0 ** -24), "rcp32": (1e-36, 1e37, True, 1.02 * 2.0 ** -24),
    "sqrt64": (1e-290, 1e290, False, 1.02 * 2.0 ** -53), "rcp64": (1e-290, 1e290, False, 1.02 * 2.0 ** -53),
    "pair_sqrt": (1e-25, 1e25, False, 2.0 ** -44), "pair_rcp": (1e-25, 1e25, False, 2.0 ** -44),
}


@pytest.mark.parametrize("fn", sorted(CASES))
def test_scalar_routine(probe, fn):
    lo, hi, single, bound = CASES[fn]
    x = _arguments(lo, hi, single)
    raw = subprocess.run([probe, fn, str(len(x))], input=x.tobytes(), check=True, capture_output=True).stdout
    got = np.frombuffer(raw, dtype=np.float64).reshape(-1, 2).astype(np.longdouble).sum(axis=1)
    if fn.startswith("pair"):        # the pair that stands for x
        h = x.astype(np.float32)
        x = h.astype(np.longdouble) + (x - h.astype(np.float64)).astype(np.float32).astype(np.longdouble)
    x = x.astype(np.longdouble)
    want = np.sqrt(x) if "sqrt" in fn else 1 / x
    err = np.abs(got - want) / want
    print(f"{fn}: largest relative error 2^{float(np.log2(err.max())):.2f}")
    assert err.max() <= bound


def test_wait_that_runs_out_names_its_kernel(probe):
    out = subprocess.run([probe, "wait", "0"], check=True, capture_output=True, text=True, timeout=60).stdout
    assert out.strip() == "2 0 an exchange of the direct split"
