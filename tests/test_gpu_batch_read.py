"""GPU tests of ts_batch_read's packed copy: jobs with fewer and more schemes
than the first copy, and than the packed entries, hold."""
import numpy as np
import pytest

import tcurve_inputs as ti

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def eng():
    import paper_2604_09221_gb300 as e
    return e


@pytest.mark.parametrize("d,counts", [
    (4, [300]), (10, [1 << 16, 70]), (13, [1000, 1024, 1500]), (16, [40, 17000, 30000])])
def test_batch_read_matches_a_sampled_sweep(eng, d, counts):
    """Every job's codes and counts against ts_enumerate of the same splitmix64
    stream (code for code), read twice."""
    tri = eng.Triangulation(d, ti.regular_triangulation(d, seed=d))
    bases = [1000 + 7 * j for j in range(len(counts))]
    batch = eng.Batch([tri] * len(counts), counts, bases, hist_capacity=1 << 16)
    batch.set_fused(True)
    batch.run()
    for j, (n, base) in enumerate(zip(counts, bases)):
        h = eng.Histogram(1 << 16, tri.code_words)
        eng.enumerate_schemes(tri, base, base + n, h, eng.TS_ENUM_SPLITMIX)
        codes, cnts, failed = h.read()
        assert failed == 0 and int(cnts.sum()) == n
        for _ in range(2):
            got, gcnt, gfailed = batch.read(j)
            assert gfailed == 0
            np.testing.assert_array_equal(got.reshape(codes.shape), codes)
            np.testing.assert_array_equal(gcnt, cnts)
