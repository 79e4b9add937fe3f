"""The bit-sliced kernels on the GPU at the edges of their blocks of 128 sign
vectors, against the oracle."""
import collections

import numpy as np
import pytest

import tcurve_inputs as ti

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def eng():
    import paper_2604_09221_gb300 as e
    return e


@pytest.mark.parametrize("d", [1, 2, 5, 8, 9, 10, 11, 16])
def test_ragged_blocks(eng, orc, d):
    """Queries and sampled sweeps of 1, 127, 128, 129 and 1000 sign vectors
    (one- and two-byte labels, twist bits in and beside the label, both back
    ends) on the fan and a regular triangulation: codes and histograms equal
    the oracle's, and nothing behind the last code is written."""
    import torch
    for edges in ([ti.fan_triangulation(d)] if d > 1 else []) + [
            ti.regular_triangulation(d, seed=500 + d) if d > 1 else ti.standard_triangulation(1)]:
        tri = eng.Triangulation(d, edges)
        otri = orc.triangles(d, edges)
        for n in (1, 127, 128, 129, 1000):
            want = orc.real_schemes(d, otri, ti.splitmix_sign_vectors(d, 77 * n, n))
            signs = eng.splitmix_masks(d, 77 * n, n)
            out = torch.full((n + 4, tri.code_words), -7, dtype=torch.int64, device="cuda")
            tri.real_schemes(signs, out=out)
            got = out.cpu().numpy()
            assert (got[:n].view(np.uint64) == want).all(), (d, n)
            assert (got[n:] == -7).all()
            h = eng.Histogram(2048, tri.code_words)
            eng.enumerate_schemes(tri, 77 * n, 77 * n + n, h, eng.TS_ENUM_SPLITMIX)
            codes, counts, failed = h.read()
            assert failed == 0
            assert ({eng.code_to_int(c): int(k) for c, k in zip(codes, counts)}
                    == dict(collections.Counter(orc.code_to_int(c) for c in want))), (d, n)
