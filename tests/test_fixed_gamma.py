"""The fixed-point kernel evaluation (csrc/fixed_gamma.cuh) against long double.

CPU part: the header compiled for the host. GPU part: the pairwise product
entry by entry, at the sizes where groups, tiles and column blocks end, and on
inputs whose dynamic range decides the path.
"""
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2101_00629_gb300", "csrc")

HOST = r"""
#define __host__
#define __device__
#define __forceinline__ inline
#include "fixed_gamma.cuh"
#include <cstdio>
#include <random>
using namespace kl;
static const fx::Exp2Table TAB;
typedef long double LD;
int main() {
    std::mt19937_64 g(1);
    LD e55 = 0, e53 = 0, dbl = 0, nrm = 0, gs = 0, fix = 0, mat = 0;
    auto up = [](LD& w, LD e) { if (!(fabsl(e) <= w)) w = fabsl(e); };
    for (int it = 0; it < 400000; ++it) {
        uint32_t n;
        uint64_t t = (g() >> 1) >> (g() % 40);
        if (it < 4096) t = (uint64_t)it << 44;           // table entries
        if (it == 5000) t = 0;
        uint64_t E = fx::exp2_neg<55>(t, TAB.v, n);
        const LD f = ldexpl((LD)t, -55);
        up(e55, ldexpl((LD)E, -63) / exp2l((LD)n - f) - 1);
        up(dbl, (LD)fx::to_double(E, n) / exp2l(-f) - 1);
        t = (g() >> 1) >> (g() % 40);
        E = fx::exp2_neg<53>(t, TAB.v, n);
        up(e53, ldexpl((LD)E, -63) / exp2l((LD)n - ldexpl((LD)t, -53)) - 1);
        uint64_t c[3];
        for (auto& v : c) v = (g() >> 2) >> (g() % 64);
        if (it % 5 == 0) c[1] = c[2] = 0;
        if (it % 7 == 0) c[1] = c[2] = c[0];
        const LD r = sqrtl((LD)c[0] * c[0] + (LD)c[1] * c[1] + (LD)c[2] * c[2]);
        up(nrm, ((LD)fx::norm3(c[0], c[1], c[2]) - r) / (1 + ldexpl(r, -58)));
        for (auto& v : c) v >>= 2;
        const LD q = ldexpl((LD)c[0] * c[0] + (LD)c[1] * c[1] + (LD)c[2] * c[2], -61);
        if (q < ldexpl(1000, 53)) up(gs, ((LD)fx::exponent<KL_KERNEL_GAUSS>(c[0], c[1], c[2]) - q) / (1 + ldexpl(q, -60)));
        t = (g() >> 2) >> (g() % 40);
        const LD m = ldexpl(1, 55) + (LD)t * 0.693147180559945309417232L;
        up(mat, ((LD)fx::matern_factor(t) - m) / (1 + ldexpl(m, -62)));
        const double x = ldexp((double)(int64_t)g(), -63 - (int)(g() % 60));
        const uint64_t sm = g() | (1ull << 63);
        up(fix, (LD)(int64_t)fx::to_fixed<55>(x, sm, -60) - ldexpl((LD)x * (LD)sm, -5));
    }
    printf("%.6Lg %.6Lg %.6Lg %.6Lg %.6Lg %.6Lg %.6Lg\n", ldexpl(e55, 53), ldexpl(e53, 53), ldexpl(dbl, 53), nrm, gs, mat, fix);
}
"""


def test_host_errors(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no g++")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(HOST)
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", CSRC, "-o", str(exe), str(src)], check=True)
    e55, e53, dbl, nrm, gs, mat, fix = map(float, subprocess.run([str(exe)], check=True, capture_output=True).stdout.split())
    # the exponential: three truncations of 2^-56 and the cubic's 2^-57.7
    assert e55 < 0.5 and e53 < 0.5
    assert dbl < 1.5            # and one rounding to 53 bits
    assert nrm < 4 and gs < 4   # units of the last place, or of 2^-58 (2^-60) of the result
    assert mat < 4
    assert fix <= 1.01          # floor (long double holds the product to 64 bits)


def _gamma(kernel, L, P, Q):
    d = [np.abs(P[j][:, None] - Q[j][None, :]) for j in range(3)]
    L = np.longdouble(L)
    if kernel == "exp_sep":
        a = (d[0] + d[1] + d[2]) / L
    elif kernel == "gauss":
        a = (d[0] ** 2 + d[1] ** 2 + d[2] ** 2) / L ** 2
    else:
        a = np.sqrt(d[0] ** 2 + d[1] ** 2 + d[2] ** 2) / L
    if kernel == "matern32":
        a = np.sqrt(np.longdouble(3)) * a
        return (1 + a) * np.exp(-a), a
    return np.exp(-a), a


@pytest.mark.gpu
@pytest.mark.parametrize("kernel", ["gauss", "exp_sep", "exp", "matern32"])
@pytest.mark.parametrize("T,S,k,L,inputs", [
    (1, 1, 1, 0.5, "normal"),
    (127, 31, 2, 2.0, "normal"),        # one ragged group, one ragged tile
    (129, 33, 3, 0.5, "normal"),
    (256, 128, 4, 0.1, "normal"),
    (300, 161, 5, 0.05, "normal"),      # values down to e^-1000
    (130, 289, 9, 0.3, "normal"),       # 16-column form
    (65, 100, 17, 1.0, "normal"),       # two passes over the columns
    (257, 96, 8, 0.1, "units"),         # columns of the kernel matrix
    (200, 320, 6, 0.3, "graded"),       # entries over 60 decades
    (150, 70, 4, 0.02, "offset"),       # far from the origin
    (140, 66, 3, 0.005, "normal"),      # beyond the fixed-point range
])
def test_pairwise_entries(kernel, T, S, k, L, inputs):
    import torch
    import paper_2101_00629_gb300 as kl
    rng = np.random.default_rng(T * 1000 + S)
    tgt, src = rng.random((3, T)), rng.random((3, S))
    n = min(T, S) // 2
    tgt[:, :n] = src[:, :n]             # coincident points
    if inputs == "offset":
        tgt, src = 1000.0 + 0.1 * tgt, 1000.0 + 0.1 * src
    X = rng.standard_normal((k, S))
    if inputs == "units":
        X = np.zeros((k, S))
        X[np.arange(k), rng.choice(S, k, replace=False)] = 1.0
    if inputs == "graded":
        X *= 10.0 ** rng.uniform(-30, 30, (k, S))
    d = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (tgt, src, X)]
    Y = torch.empty(k, T, dtype=torch.float64, device="cuda")
    kl.kl_pairwise_noalloc(kernel, 1.5, L, d[0], T, d[1], S, d[2], S, Y, T, k, torch.cuda.current_stream())
    G, a = _gamma(kernel, L, tgt.astype(np.longdouble), src.astype(np.longdouble))
    ref = 2.25 * (X.astype(np.longdouble) @ G.T)
    # what an FP64 evaluation may lose: rounding of the exponent a (a few
    # 2^-53 a), of the value, and of the sums
    bound = 2.25 * (np.abs(X).astype(np.longdouble) @ ((16 + 4 * a) * G).T) * 2.0 ** -53 + 1e-320
    assert np.all(np.abs(Y.cpu().numpy() - ref) <= bound)


@pytest.mark.gpu
@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf, 1e-310])
def test_pairwise_special_entries(bad):
    """Infinities and NaN spread as in FP64; tiny entries keep their value."""
    import torch
    import paper_2101_00629_gb300 as kl
    rng = np.random.default_rng(3)
    T, S = 140, 70
    P, Q = rng.random((3, T)), rng.random((3, S))
    X = np.zeros((2, S))
    X[0, 40] = bad
    X[1] = rng.random(S)
    d = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (P, Q, X)]
    Y = torch.empty(2, T, dtype=torch.float64, device="cuda")
    kl.kl_pairwise_noalloc("exp", 1.0, 0.7, d[0], T, d[1], S, d[2], S, Y, T, 2, torch.cuda.current_stream())
    G = _gamma("exp", 0.7, P, Q)[0].astype(np.float64)
    ref = (X[:, None, :] * G[None]).sum(2)
    np.testing.assert_allclose(Y.cpu().numpy(), ref, rtol=1e-12, atol=1e-322)


@pytest.mark.gpu
@pytest.mark.parametrize("entries", ["far", "near", "graded", "descending", "single"])
@pytest.mark.parametrize("length", [1.0, 3.0, 4.2, 5.5])
@pytest.mark.parametrize("kernel", ["exp", "gauss", "matern32", "exp_sep"])
def test_entries_of_unequal_size(kernel, length, entries):
    """Groups of 32 sources on a line, the smallest values meeting the largest
    entries: no more error than an FP64 evaluation may have. 64 groups, each the
    only one that its column has entries in."""
    import torch
    import paper_2101_00629_gb300 as kl
    n, groups, T = 32, 64, 32
    rng = np.random.default_rng(11)
    tgt, src = np.zeros((3, T)), np.zeros((3, groups * n))
    tgt[0] = 1e-3 * rng.random(T)
    pos = (np.arange(n) + rng.random((groups, n))) / n
    src[0] = 0.002 + (length * pos if kernel != "gauss" else np.sqrt(length) * pos).ravel()
    x = 1.0 + rng.random((groups, n))
    tiny = 10.0 ** -rng.uniform(8, 17, (groups, n)) * rng.choice([-1.0, 1.0], (groups, n))
    if entries == "far":
        x[:, :-1] = tiny[:, :-1]
    elif entries == "near":
        x[:, 1:] = tiny[:, 1:]
    elif entries == "graded":
        x *= 10.0 ** -rng.uniform(0, 6, (groups, n))
    elif entries == "descending":
        x *= 10.0 ** (-8.0 * np.arange(n)[::-1] / n)
    else:
        x[:, :-1] = 0.0
    X = np.zeros((groups, groups * n))
    for g in range(groups):
        X[g, g * n:(g + 1) * n] = x[g]
    d = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (tgt, src, X)]
    Y = torch.empty(groups, T, dtype=torch.float64, device="cuda")
    kl.kl_pairwise_noalloc(kernel, 1.0, 1.0, d[0], T, d[1], groups * n, d[2], groups * n, Y, T, groups,
                           torch.cuda.current_stream())
    Y = Y.cpu().numpy()
    # FP64: the exponent a from a distance with roundings of 3.5 units of 2^-53 of
    # itself, the exponential, the factor 1 + a and the product within 3 (5), and
    # one rounding for each addition that follows
    units = 5.0 if kernel == "matern32" else 3.0
    for g in range(groups):
        G, a = _gamma(kernel, 1.0, tgt.astype(np.longdouble), src[:, g * n:(g + 1) * n].astype(np.longdouble))
        xl = x[g].astype(np.longdouble)
        bound = ((units + 3.5 * a + np.arange(n)[::-1]) * G) @ np.abs(xl) * 2.0 ** -53
        assert np.all(np.abs(Y[g] - G @ xl) <= bound)
