"""Half-vector passes: cost vectors with f(x) = f(~x) are evolved on the amplitudes whose top qubit is 0.

The reference of each check is the full-vector path on the same costs, taken by clearing the mark that
cost_stats_compute leaves in `reserved`.  Tolerances: a state amplitude takes about 2 roundings per rotation, n p of
them, and 2 per phase; at 6e-8 (complex64) and n p <= 120 the root-sum-square is 1e-6 of the norm per path, so 5e-6
between two paths; complex128 the same with 1.1e-16, 1e-13 allowed.  Gradients are inner products of such vectors."""
import numpy as np
import pytest

from gpu_util import dev_np, torch
import oracle
from paper_2309_04841_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def Q():
    from paper_2309_04841_gb300 import qaoa
    return qaoa


def full(Q, s):
    return Q.CostStats(s.f_min, s.f_max, s.n_min, s.step_log2, 0)


def costs(Q, n, kind):
    """Symmetric cost vectors of every element type."""
    if kind == "i32":
        return Q.labs_costs(n)
    if kind == "u16":
        return Q.labs_costs_u16(n)
    e, w = I.maxcut_gnp(n, 0.4 if n >= 10 else 0.9, graph_seed=n, weight_seed=n + 1)
    return Q.maxcut_costs(n, e, w, Q.COST_F32 if kind == "f32" else Q.COST_F64)


def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


# n <= 13: on chip, every number of rounds and of bits in the last one.  n: every count of groups (forward 13 + 9 rows + ..., adjoint 12 + 8 or 9), a group that takes only the complement,
# odd and even numbers of index bits, groups of exactly full rows
@pytest.mark.parametrize("kind", ["i32", "u16", "f32", "f64"])
@pytest.mark.parametrize("n", [4, 5, 6, 7, 8, 9, 10, 11, 12, 13, 14, 15, 16, 17, 18, 19, 20, 21, 22, 23, 24])
def test_half_vs_full(Q, n, kind):
    T = torch()
    p = 3
    fd = costs(Q, n, kind)
    s = Q.cost_stats_compute(fd)
    assert s.reserved != 0
    g, b = I.angles(p, n, 0, 0.2), I.angles(p, 50 + n)  # betas on both sides of pi / 4: both rotation forms
    for st, tol in ((Q.C64, 5e-6), (Q.C128, 1e-13)):
        for q in (1, 2, p):  # either end of the group order ends the sweep
            a, ea = Q.simulate(fd, s, g[:q], b[:q], state_type=st)
            c, ec = Q.simulate(fd, full(Q, s), g[:q], b[:q], state_type=st)
            assert float(T.linalg.vector_norm(a - c)) < tol, (st, q)
            assert rel(dev_np(ea), dev_np(ec)) < tol
        x = T.empty(1 << n, dtype=Q.state_dtype(st), device="cuda")
        ga = dev_np(Q.grad(fd, s, g, b, state=x, state_type=st))
        gc = dev_np(Q.grad(fd, full(Q, s), g, b, state_type=st))
        assert rel(ga[:2], gc[:2]) < tol and rel(ga[2:], gc[2:]) < 10 * tol
        assert float(T.linalg.vector_norm(x - 2.0 ** (-n / 2))) < tol  # |+> again, both halves


@pytest.mark.parametrize("n", [14, 16])
def test_half_vs_oracle(Q, n):
    f = oracle.labs_costs(n).astype(float)
    fd = Q.labs_costs(n)
    s = Q.cost_stats_compute(fd)
    g, b = I.angles(3, 5, 0, 0.1), I.angles(3, 6)
    E, dg, db = oracle.grad(n, f, g, b)
    for st, tol in ((Q.C64, 1e-4), (Q.C128, 1e-9)):
        out = dev_np(Q.grad(fd, s, g, b, state_type=st))
        assert abs(out[0] - E) <= 0.1 * tol * abs(E)
        assert rel(out[2:], np.concatenate([dg, db])) < tol


def test_mark(Q):
    # one amplitude off its complement, a struct changed by hand, another n: the full path
    for n in (1, 2, 3, 5, 8, 13):
        for dt in (Q.COST_I32, Q.COST_F32, Q.COST_F64):
            fd = Q.precompute_costs(n, [(2, (0, n - 1)) if n > 1 else (2, ())], dt)
            assert Q.cost_stats_compute(fd).reserved != 0
            fd[(1 << n) - 1] += 1
            assert Q.cost_stats_compute(fd).reserved == 0
    n = 14
    fd = Q.labs_costs(n)
    s = Q.cost_stats_compute(fd)
    fd[5] += 4  # within the range and the step of the statistics
    s.f_min, s.f_max = s.f_min - 4.0, s.f_max + 4.0
    g, b = [0.05, 0.02], [0.3, 0.7]
    a, _ = Q.simulate(fd, s, g, b)
    c, _ = Q.simulate(fd, full(Q, s), g, b)
    np.testing.assert_array_equal(dev_np(a), dev_np(c))


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 7, 8, 9, 11, 12])
@pytest.mark.parametrize("st", ["c64", "c128"])
def test_on_chip_any_costs(Q, n, st):
    # no symmetry: costs with linear terms, every register tile, against the oracle; p = 130 crosses a launch
    terms = [(1, (q,)) for q in range(n)] + [(2, (0, n - 1))] * (n > 1) + [(-1, tuple(range(min(3, n))))]
    f = oracle.costs_terms_int(n, terms).astype(float)
    fd = Q.precompute_costs(n, terms)
    s = Q.cost_stats_compute(fd)
    assert s.reserved == 0 or n == 1  # (n = 1: the terms cancel)
    for p in (1, 2, 130):
        g, b = I.angles(p, n, 0, 0.3), I.angles(p, 50 + n)
        tol = (5e-6 if st == "c64" else 1e-13) * max(1.0, p / 3)
        psi = oracle.simulate(n, f, g, b)
        x, _ = Q.simulate(fd, s, g, b, state_type=Q.C64 if st == "c64" else Q.C128)
        assert np.linalg.norm(dev_np(x) - psi) < tol
        E, dg, db = oracle.grad(n, f, g, b)
        out = dev_np(Q.grad(fd, s, g, b, state_type=Q.C64 if st == "c64" else Q.C128))
        ref = np.concatenate([dg, db])
        assert np.linalg.norm(out[2:] - ref) <= 10 * tol * max(np.linalg.norm(ref), np.abs(f).max())
        assert abs(out[0] - E) <= 10 * tol * np.abs(f).max()


@pytest.mark.parametrize("n", [8, 14, 21])
def test_vector_changed_after_the_scan(Q, n):
    # what the header asks for after a write: a new scan finds the asymmetry, reserved = 0 keeps the other fields' use
    fd = Q.labs_costs(n)
    s = Q.cost_stats_compute(fd)
    fd[5] += 4  # within the range of the statistics, and but for n = 14 (steps of 8) within their step
    assert s.f_min <= float(fd[5]) <= s.f_max
    g, b = [0.05, 0.02], [0.3, 0.7]
    f = dev_np(fd).astype(float)
    ref = oracle.simulate(n, f, g, b)
    new = Q.cost_stats_compute(fd)
    assert new.reserved == 0
    s.reserved = 0
    for st in (s, new) if 4 % (1 << s.step_log2) == 0 else (new,):
        x, e = Q.simulate(fd, st, g, b, state_type=Q.C128)
        assert np.linalg.norm(dev_np(x) - ref) < 1e-13
