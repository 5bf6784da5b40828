"""Cost vectors built by the Walsh-Hadamard transform (n >= 13, sums that are exact): bit for bit the oracle's."""
import numpy as np
import pytest

import oracle
from gpu_util import dev_np
from paper_2309_04841_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def Q():
    from paper_2309_04841_gb300 import qaoa
    return qaoa


# n: one tile, two, one more than the persistent grid holds at once; 1, 1024 and 1025+ terms: chunk edges
@pytest.mark.parametrize("n,m", [(13, 1), (13, 1024), (14, 1025), (15, 2100), (21, 40)])
def test_terms(Q, n, m):
    ti = I.random_terms(n, m, 3 + n, max_order=5, integer=True, wmax=1000)
    np.testing.assert_array_equal(dev_np(Q.precompute_costs(n, ti)), oracle.costs_terms_int(n, ti).astype(np.int32))
    tr = I.random_terms(n, m, 4 + n, max_order=5, integer=False)
    f = oracle.costs_terms_real(n, tr)
    np.testing.assert_array_equal(dev_np(Q.precompute_costs(n, tr, Q.COST_F64)), f)
    if m <= 1024:
        np.testing.assert_array_equal(dev_np(Q.precompute_costs(n, tr, Q.COST_F32)), oracle.to_f32_rne(f))


@pytest.mark.parametrize("n", [13, 16])
def test_maxcut(Q, n):
    e, w = I.maxcut_gnp(n, 0.6, graph_seed=n, weight_seed=n)
    f = oracle.maxcut_costs(n, e, w)
    np.testing.assert_array_equal(dev_np(Q.maxcut_costs(n, e, w, Q.COST_F64)), f)
    np.testing.assert_array_equal(dev_np(Q.maxcut_costs(n, e, w, Q.COST_F32)), oracle.to_f32_rne(f))
    # integer weights whose doubled sum passes int32 (term by term), and just below (transform)
    for top in (2.0 ** 30, 2.0 ** 30 - 8):
        wi = np.zeros(len(e))
        wi[0], wi[-1] = top - 7, 7
        np.testing.assert_array_equal(dev_np(Q.maxcut_costs(n, e, wi)), oracle.maxcut_costs(n, e, wi).astype(np.int32))


# the transform or the loops over terms and edges (walsh_pays): either side of each count, sizes of each rule
@pytest.mark.parametrize("n", [13, 17, 18, 19, 20, 21])
@pytest.mark.parametrize("count", [1, 2, 22, 23, 32, 33, 100, 101])
def test_either_way(Q, n, count):
    terms = I.random_terms(n, count, 7 * n + count, max_order=4, integer=True)
    f = oracle.costs_terms_int(n, terms)
    for ct, dt in ((Q.COST_I32, np.int32), (Q.COST_F32, np.float32), (Q.COST_F64, np.float64)):
        np.testing.assert_array_equal(dev_np(Q.precompute_costs(n, terms, ct)), f.astype(dt))
    r = np.random.RandomState(count)
    e = r.randint(0, n, (count, 2)).astype(np.int32)
    e[:, 1] = (e[:, 0] + 1 + r.randint(0, n - 1, count)) % n
    w = np.floor(r.rand(count) * 8) + 1
    g = oracle.maxcut_costs(n, e, w)
    for ct, dt in ((Q.COST_I32, np.int32), (Q.COST_F32, np.float32), (Q.COST_F64, np.float64)):
        np.testing.assert_array_equal(dev_np(Q.maxcut_costs(n, e, w, ct)), g.astype(dt))
