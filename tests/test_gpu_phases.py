"""Every way to a phase exp(-i gamma f) of integer costs -- tables of two and three digits, computed -- against the
oracle, on chip, on the small tiles and on the streamed passes of both precisions.

Tolerances as in test_gpu_half.py: 5e-6 of the norm for complex64 states of p = 2 layers and n <= 21, 1e-13 for
complex128, ten times that for gradients.  Phases of |gamma f| <= 100 are reduced from a float pair (2^-48) or a
double pair, below both."""
import numpy as np
import pytest

from gpu_util import dev_np
import oracle
from paper_2309_04841_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def Q():
    from paper_2309_04841_gb300 import qaoa
    return qaoa


def check(Q, n, terms, scale, st, symmetric=False, u16=False, step=None):
    """Simulation and gradient of an integer polynomial at p = 2, gammas up to `scale`."""
    f = oracle.costs_terms_int(n, terms).astype(float)
    fd = Q.precompute_costs(n, terms)
    s = Q.cost_stats_compute(fd)
    assert (s.f_min, s.f_max) == (f.min(), f.max()) and (s.reserved != 0) == symmetric
    if u16:
        fd = Q.convert_costs(fd, s, Q.COST_U16)
    if step is not None:  # a struct filled by hand: 0 is always valid
        s = Q.CostStats(s.f_min, s.f_max, s.n_min, step, 0)
    g, b = I.angles(2, 5 + n, 0.2 * scale, scale), I.angles(2, 70 + n)
    tol = 5e-6 if st == Q.C64 else 1e-13
    x, e = Q.simulate(fd, s, g, b, state_type=st)
    assert np.linalg.norm(dev_np(x) - oracle.simulate(n, f, g, b)) < tol
    E, dg, db = oracle.grad(n, f, g, b)
    out = dev_np(Q.grad(fd, s, g, b, state_type=st))
    spread = np.abs(f).max()
    assert abs(out[0] - E) <= 10 * tol * spread and abs(dev_np(e)[0] - E) <= 10 * tol * spread
    for got, ref in ((out[2:4], dg), (out[4:], db)):  # d/d gamma is a factor 1 / scale the larger
        assert np.linalg.norm(got - ref) <= 10 * tol * max(np.linalg.norm(ref), spread)
    return s


# values +-2^30 +-2^29: steps of 2^30, a range of 3 2^30, so digit << shift leaves int32
@pytest.mark.parametrize("n,st", [(4, 0), (12, 0), (12, 1), (13, 0), (14, 0), (14, 1), (16, 1), (19, 0), (21, 0), (21, 1)])
@pytest.mark.parametrize("odd", [False, True])
def test_range_over_int32(Q, n, st, odd):
    terms = [(2 ** 30, (0, n - 1)), (2 ** 29, (1,) if odd else (1, 2))]
    s = check(Q, n, terms, 4e-9, st, symmetric=not odd)
    assert s.step_log2 == 30 and s.f_max - s.f_min == 3 * 2 ** 30


# complex128: at beta = 0 a layer is the phase alone, exp(-i gamma f) 2^(-n/2), here with |gamma f| up to about 430.
# The fraction of gamma f / 2 pi is known to 2^-54 of a turn (3.5e-16 in the angle), sincospi adds 2.2e-16, a table's
# product as much again for each of up to three factors: 2e-15 in all.  (With gamma / 2 pi in one double the angle is
# off by |gamma f| 2^-53 and more: 5e-14.)
# (integer costs, whose phases come from tables; a phase per amplitude takes one double, as it always did)
@pytest.mark.parametrize("n", [5, 8, 12, 14, 18, 21])
@pytest.mark.parametrize("half", [False, True])
def test_double_phase(Q, n, half):
    f = oracle.labs_costs(n)
    fd = Q.labs_costs(n)
    s = Q.cost_stats_compute(fd)
    if not half:
        s.reserved = 0
    gamma = 430.1 / f.max()
    x, _ = Q.simulate(fd, s, [gamma], [0.0], state_type=Q.C128)
    v, at = np.unique(f, return_inverse=True)
    a = np.longdouble(gamma) * v.astype(np.longdouble)
    ref = (np.cos(a).astype(float) - 1j * np.sin(a).astype(float))[at.reshape(-1)]
    assert np.abs(dev_np(x) * 2.0 ** (n / 2) - ref).max() < 2e-15


# Costs so large that even the low part of gamma f / 2 pi, a float pair, is many turns: the phase carries no
# information then, but every factor still has modulus one, and the amplitudes of the costs beside them are exact.
@pytest.mark.parametrize("n", [12, 14, 21, 22])
@pytest.mark.parametrize("half", [False, True])
def test_penalty_costs(Q, n, half):
    import torch
    f = Q.labs_costs(n).float()
    big = torch.logspace(10, 35, f[5::64].numel(), dtype=torch.float64).float()
    f[5::64] = big.to(f.device)
    if half:
        f = torch.maximum(f, f.flip(0))
    s = Q.cost_stats_compute(f)
    assert (s.reserved != 0) == half
    x, _ = Q.simulate(f, s, [0.31], [0.0], state_type=Q.C64)
    x = dev_np(x) * 2.0 ** (n / 2)
    f0 = dev_np(f).astype(float)
    assert np.abs(np.abs(x) - 1.0).max() < 2e-6  # the phase's and the scale's roundings
    assert np.abs(x - np.exp(-1j * 0.31 * f0))[f0 < 1e6].max() < 2e-6
    x, _ = Q.simulate(f, s, [0.31, 0.23], [0.4, 0.2], state_type=Q.C64)
    assert abs(float(torch.linalg.vector_norm(x)) - 1.0) < 5e-6


# complex64 tables: with beta = 0 a layer multiplies every amplitude by the same table product, so 32 equal layers add an
# entry's error up 32 times.  Entries within 0.55 ulp (2.4e-8 rms a complex entry below one) and one product of two
# (3.4e-8): 32 sqrt(2 * 2.4^2 + 3.4^2) e-8 = 1.5e-6 rms; with the angle rounded to float before its sine and cosine an
# entry has 4e-8 more and the sum is above 2e-6 for some gammas.  1.6e-6 allowed on the mean of four gammas.
@pytest.mark.parametrize("n", [13, 14, 16, 18, 19])
@pytest.mark.parametrize("half", [False, True])
def test_single_table_entries(Q, n, half):
    f, fd, p = oracle.labs_costs(n), Q.labs_costs(n), 32
    s = Q.cost_stats_compute(fd)
    if not half:
        s.reserved = 0
    rms = []
    for gamma in (0.013, 0.0371, 0.077, 0.1):
        x, _ = Q.simulate(fd, s, [gamma] * p, [0.0] * p, state_type=Q.C64)
        d = dev_np(x) * 2.0 ** (n / 2) - np.exp(-1j * gamma * p * f)
        rms.append(np.sqrt(np.mean(np.abs(d) ** 2)))
    assert np.mean(rms) < 1.6e-6


# weights, and the number of steps of the cost's range: tables of two digits take up to 3071 (streamed complex64) or
# 8191 steps, of three up to 32767 or 262143, larger ranges are computed (n <= 12: tables up to 8191, then computed)
WAYS = {"two": ((400, 148, 12), 140), "three": ((4001, 1503, 7), 5511), "three_wide": ((15001, 12503, 7), 27511),
        "three_most": ((120001, 110003, 7), 230011), "computed": ((300001, 250003, 7), 550011)}


@pytest.mark.parametrize("n,st", [(12, 0), (12, 1), (13, 0), (16, 0), (16, 1), (21, 0), (21, 1), (22, 0)])
@pytest.mark.parametrize("way", list(WAYS))
@pytest.mark.parametrize("half", [False, True])
def test_every_way(Q, n, st, way, half):
    (a, b, c), steps = WAYS[way]
    terms = [(a, (0, n - 1)), (b, (2, 5) if half else (2,)), (c, (3, 4))] + [(c, (3, 4, 6))] * (not half)
    s = check(Q, n, terms, 100.0 / (a + b + 2 * c), st, symmetric=half)
    assert abs((s.f_max - s.f_min) / 2 ** s.step_log2 - steps) <= 14


# uint16 costs: differences are even, so 32767 steps are the most; step_log2 = 0 by hand leaves tables of three digits
@pytest.mark.parametrize("n,st", [(13, 0), (16, 1), (21, 0), (21, 1)])
@pytest.mark.parametrize("step", [None, 0])
def test_uint16_ways(Q, n, st, step):
    for (a, b, c) in ((400, 148, 12), (4001, 1503, 7), (15001, 12503, 7)):
        terms = [(a, (0, n - 1)), (b, (2,)), (c, (3, 4)), (a + b + c, ())]
        check(Q, n, terms, 100.0 / (2 * (a + b + c)), st, u16=True, step=step)


# float32 costs on the streamed passes: table entry (2.4e-8 rms), sine and cosine of the rest (1.7e-8) and their product
# (2.4e-8) repeat in each of 32 equal layers, 32 * 3.8e-8 = 1.2e-6; with the fraction of gamma f / 2 pi rounded to one
# float (5e-8 where it is above a quarter turn) 1.8e-6.  1.4e-6 allowed on the mean of four gammas.
@pytest.mark.parametrize("n", [21, 22])
@pytest.mark.parametrize("kind", ["labs", "gnp"])
def test_float_phases(Q, n, kind):
    p = 32
    if kind == "labs":
        fd, gammas = Q.labs_costs(n).float(), (0.013, 0.0371, 0.077, 0.1)
    else:
        e, w = I.maxcut_gnp(n, 0.5, graph_seed=3, weight_seed=4)
        fd, gammas = Q.maxcut_costs(n, e, w, Q.COST_F32), (0.11, 0.23, 0.37, 0.6)
    s = Q.cost_stats_compute(fd)
    f, rms = dev_np(fd).astype(float), []
    for gamma in gammas:
        x, _ = Q.simulate(fd, s, [gamma] * p, [0.0] * p, state_type=Q.C64)
        d = dev_np(x) * 2.0 ** (n / 2) - np.exp(-1j * gamma * p * f)
        rms.append(np.sqrt(np.mean(np.abs(d) ** 2)))
    assert np.mean(rms) < 1.4e-6
