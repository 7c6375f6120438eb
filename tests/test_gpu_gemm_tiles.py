"""GPU: the grouped product kernel at the edges of its output tiles (16, 32, 64
square; slices of 8 to 32 along k), one problem and several, through a merge
and a projection: an identity cluster unitary, nothing discarded, so the state
afterwards contracts to what was loaded.

Tolerance: two products and one orthogonal basis, each with a backward error of
a few eps sqrt(n): 8 eps sqrt(n)."""
import numpy as np
import pytest

from gpu_helpers import lib

pytestmark = pytest.mark.gpu


# (chi_L, chi_mid, chi_R) of the clusters of one step; the last ones fill the chip with 32 and with 64 wide tiles
STEPS = [[(1, 1, 1)], [(8, 7, 9)], [(8, 9, 8), (17, 33, 16)], [(31, 15, 33)], [(64, 65, 63)] * 3,
         [(200, 31, 190)] * 2, [(420, 64, 410)]]


@pytest.mark.parametrize("prec", ["FP32", "FP64"])
@pytest.mark.parametrize("shapes", STEPS)
def test_products_at_tile_edges(shapes, prec):
    P = lib()
    rng = np.random.default_rng(len(shapes) + shapes[0][0])
    chis, sites = [1], []
    for a, b, c in shapes:
        for x, y in ((1, a), (a, b), (b, c), (c, 1)):
            g = rng.standard_normal((x, 2, y)) + 1j * rng.standard_normal((x, 2, y))
            sites.append((g / np.linalg.norm(g)).astype(np.complex64 if prec == "FP32" else np.complex128))
            chis.append(y)
    lams = [np.full(c, c ** -0.5) for c in chis]
    big = 2 * max(chis)
    lg = int(np.ceil(np.log2(max(big, 2))))
    mps = P.MPS(P.make_config(len(sites), big, 0.0, 2 + 2 * lg, 0, 2, getattr(P, prec)))
    mps.load(np.array(chis, dtype=np.int32), sites, lams)
    f = mps.step([P.Cluster(1 + 4 * i, 2, 0, 0) for i in range(len(shapes))], [np.eye(4, dtype=np.complex128)] * len(shapes))
    eps = 2.0 ** -23 if prec == "FP32" else 2.0 ** -52
    for i, (a, b, c) in enumerate(shapes):
        q = 1 + 4 * i
        tol = 8 * eps * np.sqrt(2 * max(a, b, c))
        r = int(mps.bond_dims()[q + 1])
        want = sites[q].astype(np.complex128).reshape(2 * a, b) @ sites[q + 1].astype(np.complex128).reshape(b, 2 * c)
        have = mps.site(q).reshape(2 * a, r) @ mps.site(q + 1).reshape(r, 2 * c)
        assert r == min(2 * a, b, 2 * c), (a, b, c, r)
        assert np.linalg.norm(have / np.linalg.norm(have) - want / np.linalg.norm(want)) <= tol
        assert abs(f[i] - 1) <= tol
