"""The fixed-point collision of the FP64 kernels (fixed.cuh), compiled for the host.

The same source is compared with the collision in long double and with it in double, over
random nodes: its error may not be larger than the double arithmetic's, in the mean and at
most, per population relative to that population's equilibrium (so that trace species
count), on every lattice shape it serves, both relaxation modes, and from strong to weak
departures from equilibrium.  Each species' mass is carried over up to the rounding of one
population.  Nodes that do not fit are refused and left as they were.
"""

import ctypes
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)

SOURCE = r"""
#include "fixed.cuh"
using namespace lbms;
#define LATTICE(NAME, q, np, k0, expr, c) \
    struct NAME { static constexpr int Q = q, NPAIR = np, K0 = k0; \
                  static constexpr double w(int k) { return expr; } static constexpr double cs2() { return c; } }
LATTICE(D1Q3, 3, 1, 1, k == 0 ? 2.0 / 3.0 : 1.0 / 6.0, 1.0 / 3.0);
LATTICE(D2Q4, 4, 2, 0, 0.25, 0.5);
LATTICE(D2Q5, 5, 2, 1, k == 0 ? 1.0 / 3.0 : 1.0 / 6.0, 1.0 / 3.0);
LATTICE(D2Q9, 9, 4, 1, k == 0 ? 4.0 / 9.0 : (k < 5 ? 1.0 / 9.0 : 1.0 / 36.0), 1.0 / 3.0);
LATTICE(D3Q6, 6, 3, 0, 1.0 / 6.0, 1.0 / 3.0);
LATTICE(D3Q7, 7, 3, 1, k == 0 ? 0.25 : 0.125, 0.25);
LATTICE(D3Q15, 15, 7, 1, k == 0 ? 2.0 / 9.0 : (k < 7 ? 1.0 / 9.0 : 1.0 / 72.0), 1.0 / 3.0);

template <typename L, int S, typename T>
void plain(const double* in, T* out, const double (&invD)[LBMS_MAX_SPECIES][LBMS_MAX_SPECIES], int srt)
{
    const T k = T(1) / T(L::cs2());
    T f[S][L::Q], x[S + 1], K[S][S], M[S][S], E[S][S];
    T left = T(1);
    for (int s = 0; s < S; ++s) {
        x[s] = 0;
        for (int q = 0; q < L::Q; ++q) { f[s][q] = in[s * L::Q + q]; x[s] += f[s][q]; }
        left -= x[s];
    }
    x[S] = left;
    for (int i = 0; i < S; ++i)
        for (int j = 0; j < S; ++j) {
            T b = 0;
            if (i != j) b = x[i] * (T(invD[i][S]) - T(invD[i][j]));
            else { b = x[i] * T(invD[i][S]); for (int m = 0; m <= S; ++m) if (m != i) b += x[m] * T(invD[i][m]); }
            M[i][j] = b / 2;
            K[i][j] = b / 2 + (i == j ? k : T(0));
        }
    for (int p = 0; p < S; ++p) {
        const T inv = T(1) / K[p][p];
        for (int j = 0; j < S; ++j) { K[p][j] *= inv; M[p][j] *= inv; }
        for (int r = 0; r < S; ++r) {
            if (r == p) continue;
            const T c = K[r][p];
            for (int j = 0; j < S; ++j) { K[r][j] -= c * K[p][j]; M[r][j] -= c * M[p][j]; }
        }
    }
    for (int i = 0; i < S; ++i)
        for (int j = 0; j < S; ++j) E[i][j] = !srt && i == j ? 4 * (M[i][i] - 1) / (M[i][i] - 4) : M[i][j];
    T moved[S];
    for (int s = 0; s < S; ++s) moved[s] = 0;
    for (int pr = 0; pr < L::NPAIR; ++pr) {
        const int a = L::K0 + 2 * pr, b = a + 1;
        for (int i = 0; i < S; ++i) {
            T e = 0, o = 0;
            for (int j = 0; j < S; ++j) {
                e += E[i][j] * (f[j][a] + f[j][b] - 2 * T(L::w(a)) * x[j]);
                o += M[i][j] * (f[j][a] - f[j][b]);
            }
            out[i * L::Q + a] = f[i][a] - (e + o);
            out[i * L::Q + b] = f[i][b] - (e - o);
            if (a != 0) moved[i] += f[i][a] - out[i * L::Q + a];
            moved[i] += f[i][b] - out[i * L::Q + b];
        }
    }
    for (int s = 0; s < S; ++s) out[s * L::Q] = f[s][0] + moved[s];
}

template <typename L, int S>
int run(int nodes, const double* in, const double* invD, int srt, double* fixed, double* error, double* error_double,
        double* mass, int* fits)
{
    double inv[LBMS_MAX_SPECIES][LBMS_MAX_SPECIES] = {};
    for (int i = 0; i <= S; ++i) for (int j = 0; j <= S; ++j) inv[i][j] = invD[i * (S + 1) + j];
    const FixedTable t = fixed_table(S + 1, inv, L::cs2(), srt ? LBMS_RELAX_SRT : LBMS_RELAX_MAGIC);
    if (!t.on) return 0;
    constexpr int N = S * L::Q;
    for (int n = 0; n < nodes; ++n) {
        double f[S][L::Q], d[N];
        long double e[N];
        memcpy(f, in + n * N, sizeof(f));
        fits[n] = collide_fixed<L, S>(f, t);
        memcpy(fixed + n * N, f, sizeof(f));
        plain<L, S, long double>(in + n * N, e, inv, srt);
        plain<L, S, double>(in + n * N, d, inv, srt);
        for (int q = 0; q < N; ++q) {
            error[n * N + q] = (double)(fixed[n * N + q] - e[q]);
            error_double[n * N + q] = (double)(d[q] - e[q]);
        }
        for (int s = 0; s < S; ++s) {
            long double a = 0;
            for (int q = 0; q < L::Q; ++q) a += (long double)f[s][q] - (long double)in[n * N + s * L::Q + q];
            mass[n * S + s] = (double)a;
        }
    }
    return 1;
}
#define ENTRY(NAME) \
    extern "C" int run_##NAME(int S, int nodes, const double* in, const double* invD, int srt, double* fixed, double* error, \
                              double* error_double, double* mass, int* fits) { \
        return S == 1 ? run<NAME, 1>(nodes, in, invD, srt, fixed, error, error_double, mass, fits) \
                      : run<NAME, 2>(nodes, in, invD, srt, fixed, error, error_double, mass, fits); }
ENTRY(D1Q3) ENTRY(D2Q4) ENTRY(D2Q5) ENTRY(D2Q9) ENTRY(D3Q6) ENTRY(D3Q7) ENTRY(D3Q15)
"""

WEIGHTS = {
    "D1Q3": [2 / 3] + [1 / 6] * 2, "D2Q4": [1 / 4] * 4, "D2Q5": [1 / 3] + [1 / 6] * 4,
    "D2Q9": [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4, "D3Q6": [1 / 6] * 6, "D3Q7": [1 / 4] + [1 / 8] * 6,
    "D3Q15": [2 / 9] + [1 / 9] * 6 + [1 / 72] * 8,
}
CS2 = {"D1Q3": 1 / 3, "D2Q4": 1 / 2, "D2Q5": 1 / 3, "D2Q9": 1 / 3, "D3Q6": 1 / 3, "D3Q7": 1 / 4, "D3Q15": 1 / 3}


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("fixed")
    src, so = str(d / "fixed.cpp"), str(d / "fixed.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.run(["g++", "-O2", "-std=c++17", "-w", "-shared", "-fPIC", "-ffp-contract=off",
                    "-I", os.path.join(ROOT, "paper_1808_06787_gb300", "csrc"), "-I", os.path.join(ROOT, "include"),
                    src, "-o", so], check=True)
    return ctypes.CDLL(so)


def collide(lib, lattice, S, f, D, srt):
    nodes = f.shape[0]
    Q = len(WEIGHTS[lattice])
    f = np.ascontiguousarray(f, dtype=np.float64).reshape(nodes, S * Q)
    inv = np.ascontiguousarray(1.0 / D)
    out, err, errd = (np.empty_like(f) for _ in range(3))
    mass, fits = np.empty((nodes, S)), np.empty(nodes, dtype=np.int32)
    p = lambda a: a.ctypes.data_as(ctypes.c_void_p)  # noqa: E731
    on = getattr(lib, "run_" + lattice)(S, nodes, p(f), p(inv), srt, p(out), p(err), p(errd), p(mass), p(fits))
    shape = (nodes, S, Q)
    return on, out.reshape(shape), err.reshape(shape), errd.reshape(shape), mass, fits.astype(bool)


def nodes_of(lattice, S, count, amp, kind, g):
    w = np.array(WEIGHTS[lattice])
    x = g.uniform(0.0, 1.0, (count, S + 1)) + 1e-3
    if kind == "trace":
        x[:, 0] *= 10.0 ** g.uniform(-30, -3, count)
    if kind == "absent":
        x[:, 0] = 0.0
    x /= x.sum(1, keepdims=True)
    f = w * x[:, :S, None] * (1.0 + amp * g.uniform(-0.5, 0.5, (count, S, w.size)))
    return f, x


def matrix(n, g, lo=0.01, hi=0.12):
    D = np.ones((n, n))
    for i in range(n):
        for j in range(i + 1, n):
            D[i, j] = D[j, i] = g.uniform(lo, hi)
    return D


@pytest.mark.parametrize("srt", [0, 1])
@pytest.mark.parametrize("kind", ["plain", "trace", "absent"])
@pytest.mark.parametrize("S", [1, 2])
@pytest.mark.parametrize("lattice", sorted(WEIGHTS))
def test_no_larger_error_than_double(lib, lattice, S, kind, srt):
    g = np.random.default_rng([len(lattice), S, len(kind), srt, len(WEIGHTS[lattice])])
    w = np.array(WEIGHTS[lattice])
    mine, double, taken = [], [], []
    for amp in (0.4, 1e-2, 1e-6):
        for _ in range(4):
            D = matrix(S + 1, g)
            f, x = nodes_of(lattice, S, 1500, amp, kind, g)
            on, out, err, errd, mass, fits = collide(lib, lattice, S, f, D, srt)
            assert on
            taken.append(fits.mean())
            scale = np.where(x[:, :S, None] > 0, w * x[:, :S, None], 1.0)[fits]
            mine.append(err[fits] / scale)
            double.append(errd[fits] / scale)
            # every result: its own rounding, and four units of the block (2^-58 of the power of
            # two above the largest population, so at most 2^-57 of the largest): the two
            # products and the equilibrium rounded to half a unit each, a unit for the rest;
            # and the other species' departures, taken in units of 2^-58 of one, through
            # Lambda_12 = G xi_1 (twice: even and odd)
            biggest = np.abs(f[fits]).max(2, keepdims=True)
            bound = np.spacing(np.abs(out[fits])) / 2 + 4 * 2.0 ** -57 * biggest
            if S == 2:
                k = 1.0 / CS2[lattice]
                a, b, c = 0.5 / D[0, 2], 0.5 / D[1, 2], 0.5 / D[0, 1]
                low = min((a + k) * (b + k), (a + k) * (c + k), (b + k) * (c + k))
                G = k * np.array([abs(a - c), abs(b - c)]) / low
                bound = bound + 2 * 2.0 ** -58 * G[:, None] * x[fits][:, :2, None]
            moving = slice(1, None)
            assert (np.abs(err[fits]) <= bound)[:, :, moving].all()
            # the mass: one rounding of population 0, and half a unit per population converted
            whole = np.abs(out[fits][:, :, 0])
            assert (np.abs(mass[fits]) <= np.spacing(whole) / 2 + w.size * 2.0 ** -58 * biggest[:, :, 0]).all()
    assert np.mean(taken) > 0.9
    # over the departures together: at the weakest both arithmetics do little more than round
    # their results, and differ by a few per cent either way
    mine, double = np.concatenate(mine), np.concatenate(double)
    assert np.sqrt((mine ** 2).mean()) <= np.sqrt((double ** 2).mean())
    assert np.abs(mine).max() <= np.abs(double).max()


def test_refused_nodes_stay(lib):
    g = np.random.default_rng(3)
    D = matrix(3, g)
    f, _ = nodes_of("D2Q5", 2, 12, 0.1, "plain", g)
    f[0, 0, 0] = np.nan
    f[1, 1, 3] = np.inf
    f[2, 0, 1] = 1.0
    f[3, 0, 1] += 0.9
    f[4] *= -1.0
    f[5, 0, 2] = -1e300
    f[6, 0] *= 1e-290
    f[7, 0] = 0.0
    f[8, 0, 1:] = 5e-324
    f[9, 0] = -0.0
    on, out, _, _, _, fits = collide(lib, "D2Q5", 2, f, D, 0)
    assert on and list(fits[:7]) == [False] * 7
    assert np.array_equal(out[:7], f[:7], equal_nan=True)
    assert fits[7] and fits[9] and not out[7, 0].any() and not out[9, 0].any()
    assert fits[10] and fits[11]


@pytest.mark.parametrize("pairs,applies", [
    ((0.1, 0.08, 0.02), True), ((0.01, 0.12, 0.12), True), ((0.833, 0.833, 0.168), True), ((0.1, 0.1, 0.1), True),
    ((1e-4, 0.1, 0.1), False), ((10.0, 10.0, 10.0), False), ((0.1, 5.0, 0.1), False)])
def test_range_of_the_diffusivities(lib, pairs, applies):
    D = np.ones((3, 3))
    D[0, 1] = D[1, 0] = pairs[0]
    D[0, 2] = D[2, 0] = pairs[1]
    D[1, 2] = D[2, 1] = pairs[2]
    f, _ = nodes_of("D2Q5", 2, 4, 0.1, "plain", np.random.default_rng(1))
    assert bool(collide(lib, "D2Q5", 2, f, D, 0)[0]) == applies


def wild_nodes(lattice, S, count, g):
    """Nodes far from equilibrium: moving populations of either sign from 1e-3 to one in
    magnitude, species by species, with mole fractions in [-1/16, 17/16] (population 0 takes
    what is left), among them trace species beside a wild one."""
    Q = len(WEIGHTS[lattice])
    amp = 10.0 ** g.uniform(-3, 0, (count, S, 1))
    f = amp * g.uniform(-1.0, 1.0, (count, S, Q))
    x = g.uniform(-0.05, 1.05, (count, S))
    f[:, :, 0] = x - f[:, :, 1:].sum(2)
    calm = np.array(WEIGHTS[lattice]) * x[:, :, None]
    pick = g.integers(0, 4, count)
    for s in range(S):
        f[pick == s, s] = calm[pick == s, s]  # one species at equilibrium
    trace = pick == 3
    f[trace, 0] *= 10.0 ** g.uniform(-30, -3, (trace.sum(), 1))
    if Q in (5, 7, 9, 15):  # opposite pairs that cancel in the sum, one of them large
        for i in range(0, count, 5):
            b = g.uniform(0.3, 0.9999)
            f[i, 0, 1:5] = [b, b, -b, -b]
            f[i, 0, 5:] *= 0.05
            f[i, 0, 0] = g.uniform(0.0, 0.9) - f[i, 0, 1:].sum()
    return f


@pytest.mark.parametrize("srt", [0, 1])
@pytest.mark.parametrize("S", [1, 2])
@pytest.mark.parametrize("lattice", sorted(WEIGHTS))
def test_wild_nodes_are_right_or_refused(lib, lattice, S, srt):
    """Whatever node is taken comes out right to 2^-47 of the species' largest population
    before or after: the coefficients' errors are at most some 2^-50 of the departures they
    multiply, for diffusivities within a factor of twelve.  A number that does not fit
    its field is wrong by orders of magnitude more."""
    g = np.random.default_rng([7, len(lattice), S, srt, len(WEIGHTS[lattice])])
    taken = 0
    for _ in range(4):
        f = wild_nodes(lattice, S, 20000, g)
        on, out, err, _, mass, fits = collide(lib, lattice, S, f, matrix(S + 1, g), srt)
        assert on
        assert np.array_equal(out[~fits], f[~fits])
        scale = np.maximum(np.abs(f).max(2), np.abs(out).max(2))
        assert (np.abs(err[fits]).max(2) <= 2.0 ** -47 * scale[fits]).all()
        assert (np.abs(mass[fits]) <= 2.0 ** -47 * scale[fits]).all()
        taken += fits.sum()
    assert taken > 2000


@pytest.mark.parametrize("S", [1, 2])
@pytest.mark.parametrize("lattice", sorted(WEIGHTS))
def test_subnormal_species_are_refused(lib, lattice, S):
    """A species whose populations are all subnormal has a block exponent of zero without
    being zero: it has to go to the FP64 arithmetic, not to zero."""
    g = np.random.default_rng(11)
    f, _ = nodes_of(lattice, S, 8, 0.1, "plain", g)
    Q = f.shape[2]
    f[:4, 0] = 0.0
    f[0, 0] = 5e-324
    f[1, 0] = -1e-310
    f[2, 0, Q - 1] = 2e-308
    f[3, 0, 0] = 1e-320
    f[4, 0] = 0.0  # exactly absent
    f[5, 0] = -0.0
    on, out, _, _, _, fits = collide(lib, lattice, S, f, matrix(S + 1, g), 0)
    assert on and list(fits) == [False] * 4 + [True] * 4
    assert np.array_equal(out[:4], f[:4])
    assert not out[4:6, 0].any()
