"""FP64 pairwise products of points many correlation lengths apart: every value
to its own size, wherever the kernel's exponent lies in the range of the
fixed-point evaluation or beyond it (a sum over near and far pairs would hide
the far ones). Against long double: the evaluation compiled for the host, and
the product on the GPU."""
import os
import shutil
import subprocess

import numpy as np
import pytest

from oracle import galerkin
from oracle.problem import Problem

LN2 = np.log(2.0)


def _exponent(kernel, L, d):
    """-log of the kernel's exponential factor in long double; d: (3, ...)."""
    L = np.longdouble(L)
    d = np.abs(d.astype(np.longdouble))
    if kernel == "exp_sep":
        return d.sum(0) / L
    if kernel == "gauss":
        return (d ** 2).sum(0) / L ** 2
    a = np.sqrt((d ** 2).sum(0)) / L
    return np.sqrt(np.longdouble(3)) * a if kernel == "matern32" else a


def _product(kernel, L, tgt, src, X):
    import torch
    import paper_2101_00629_gb300 as kl
    d = [torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).cuda() for a in (tgt, src, X)]
    T, S, k = tgt.shape[1], src.shape[1], X.shape[0]
    Y = torch.empty(k, T, dtype=torch.float64, device="cuda")
    kl.kl_pairwise_noalloc(kernel, 1.0, L, d[0], T, d[1], S, d[2], S, Y, T, k, torch.cuda.current_stream())
    return Y.cpu().numpy()


def _check(kernel, L, tgt, src, X):
    Y = _product(kernel, L, tgt, src, X)
    a = _exponent(kernel, L, tgt[:, :, None] - src[:, None, :])
    G = np.exp(-a) * (1 + a if kernel == "matern32" else 1)
    Xl = X.astype(np.longdouble)
    ref = Xl @ G.T
    # what an FP64 evaluation may lose: rounding of the exponent a (a few
    # 2^-53 a), of the value and of the sum; one unit of the subnormal range
    # per term
    bound = np.abs(Xl) @ ((16 + 4 * a) * G).T * 2.0 ** -53 + src.shape[1] * 2.0 ** -1073
    assert np.all(np.isfinite(Y))
    assert np.all(np.abs(Y - ref) <= bound)


@pytest.mark.gpu
@pytest.mark.parametrize("entry", [1.0, -1e-30, 1e-60, 1e-95])
@pytest.mark.parametrize("base", [600, 700, 767, 768, 900, 966, 967, 968, 985, 999])
def test_gaussian_group_scale(base, entry):
    """Groups that are narrow far away: a single point, a compact group of 32,
    and a group of one point behind a full one."""
    r = np.sqrt((base + np.linspace(0.0, 0.9, 5)) * LN2)
    tgt = np.zeros((3, 5))
    tgt[0] = r
    for S in (1, 32, 33):
        src = np.zeros((3, S))
        src[1] = 0.01 * np.arange(S) / 32
        X = np.zeros((2, S))
        X[0, -1] = entry
        X[1] = entry * (1.0 + np.arange(S) / 64)
        for t in range(5):  # one target at a time: a warp takes one path
            _check("gauss", 1.0, tgt[:, t:t + 1], src, X)


@pytest.mark.gpu
@pytest.mark.parametrize("geometry,L", [("cube", 0.066), ("cube", 0.05), ("annulus", 0.115), ("annulus", 0.105)])
def test_gaussian_operator_of_short_length(geometry, L):
    """Corner groups of a grid with 4 m + 1 points hold one point and are narrow
    at any distance."""
    import torch
    import paper_2101_00629_gb300 as kl
    prob = Problem(geometry, 2, (7, 7, 7), "gauss", 1.0, L)
    A, _, parts = galerkin.matrices(prob, with_parts=True)
    Q = np.linalg.solve(parts["Bt"].T, parts["M"])
    absA = np.abs(Q).T @ (parts["J"][:, None] * parts["Gamma"] * parts["J"][None, :]) @ np.abs(Q)
    h = kl.kl_create(kl.params(geometry=geometry, degree=2, elems=(7, 7, 7), kernel="gauss", L=L, method="galerkin",
                               precision="fp64"), torch.cuda.current_stream())
    try:
        N, _, _ = kl.kl_dims(h)
        X = np.random.default_rng(5).standard_normal((3, N))
        Xd = torch.from_numpy(X).cuda()
        Y = torch.empty_like(Xd)
        kl.kl_apply_A(h, Xd, N, Y, N, 3)
        err = np.abs(Y.cpu().numpy() - (A @ X.T).T)
        assert np.all(err <= 1e-12 * (absA @ np.abs(X).T).T)
    finally:
        kl.kl_destroy(h)


@pytest.mark.gpu
@pytest.mark.parametrize("L", [1e-320, 1e-310, 1e-300, 1e-160, 1e-100, 1e100, 1e200, 1e300])
@pytest.mark.parametrize("kernel", ["gauss", "exp_sep", "exp", "matern32"])
def test_extreme_lengths(kernel, L):
    """Lengths whose inverse (or its square) leaves the FP64 range: what the
    FP64 formula gives, NaN at coincident points among it."""
    x = np.array([0.0, 1e-310, 1e-160, 1e-20, 1.0, 1e30])
    Y = np.zeros(6)
    for t in range(6):  # one target at a time: a warp takes one path
        Y[t] = _product(kernel, L, np.array([[x[t]], [0.0], [0.0]]), np.zeros((3, 1)), np.ones((1, 1)))[0, 0]
    with np.errstate(all="ignore"):
        inv = np.float64(1.0) / np.float64(L * L) if kernel == "gauss" else np.float64(1.0) / np.float64(L)
        if kernel == "matern32":
            inv = np.sqrt(3.0) / np.float64(L)
        s = inv * (x * x if kernel == "gauss" else np.sqrt(x * x) if kernel != "exp_sep" else x)
        ref = np.exp(-s) * (1 + s if kernel == "matern32" else 1)
    np.testing.assert_allclose(Y, ref, rtol=1e-12, atol=1e-322)


HOST = r"""
#define __host__
#define __device__
#define __forceinline__ inline
#include "fixed_gamma.cuh"
#include <cstdio>
using namespace kl;
static const fx::Exp2Table TAB;
typedef long double LD;
// largest error of 2^-t, in units of 2^-53 of itself, for differences along one
// direction and along the diagonal up to the largest exponent of the format
template <int K> LD worst() {
    LD w = 0;
    const LD one = ldexpl(1, fx::Format<K>::kCoord);
    for (int diag = 0; diag < 2; ++diag)
        for (int i = 1; i <= 4000; ++i) {
            const LD t = fx::Format<K>::kMaxArg * (LD)i / 4000;
            const LD share = K == KL_KERNEL_EXP_SEP ? t / 3 : sqrtl((K == KL_KERNEL_GAUSS ? t : t * t) / 3);
            const LD d = diag ? share : (K == KL_KERNEL_GAUSS ? sqrtl(t) : t);
            const uint64_t u = (uint64_t)(d * one);
            for (int back = 0; back < 2; ++back) {
                const uint64_t x = fx::absdiff(back ? 0 : u, back ? u : 0), y = diag ? x : 0;
                uint32_t n;
                const uint64_t e = fx::exponent<K>(x, y, y);
                const uint64_t E = fx::exp2_neg<fx::Format<K>::kArg>(e, TAB.v, n);
                const LD c = (LD)u / one;
                const LD q = K == KL_KERNEL_GAUSS ? c * c * (diag ? 3 : 1) : diag ? (K == KL_KERNEL_EXP_SEP ? 3 * c : c * sqrtl(3)) : c;
                const LD r = fabsl(ldexpl((LD)E, -63) * exp2l(-(LD)n) / exp2l(-q) - 1) * ldexpl(1, 53);
                if (!(r <= w)) w = r;
            }
        }
    return w;
}
int main() {
    printf("%.6Lg %.6Lg %.6Lg\n", worst<KL_KERNEL_GAUSS>(), worst<KL_KERNEL_EXP_SEP>(), worst<KL_KERNEL_EXP>());
    return 0;
}
"""


def test_host_full_range(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no g++")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(HOST)
    csrc = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2101_00629_gb300", "csrc")
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", csrc, "-o", str(exe), str(src)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True).stdout.split()
    # the exponential (below 0.5), and the exponent: one unit of 2^-55 (2^-53)
    # per difference and one of the result, times ln 2; the reference's own
    # exponent carries 64 bits of a number below 2^10
    assert all(float(e) < 0.5 + 4 + 1 for e in out)


@pytest.mark.gpu
@pytest.mark.parametrize("S", [1, 32])
@pytest.mark.parametrize("along", ["axis", "diagonal"])
@pytest.mark.parametrize("kernel,most", [("gauss", 1000), ("exp_sep", 500), ("exp", 120), ("matern32", 120)])
def test_every_exponent(kernel, most, along, S):
    """One point and one compact group against targets at exponents (base 2)
    from 0 to beyond the fixed-point range."""
    T, L = 700, 0.5
    t = np.linspace(0.0, 1.1 * most, T)
    direction = np.array([1.0, 0.0, 0.0]) if along == "axis" else np.ones(3)
    unit = direction.sum() if kernel == "exp_sep" else np.sqrt((direction ** 2).sum())
    r = L * (np.sqrt(t * LN2) if kernel == "gauss" else t * LN2 / (np.sqrt(3) if kernel == "matern32" else 1)) / unit
    tgt = 0.25 + direction[:, None] * r
    src = np.full((3, S), 0.25)
    src[1] += 0.003 * np.arange(S) / 32
    src[2] += 0.002 * (np.arange(S) % 4)
    X = np.random.default_rng(1).uniform(0.5, 1.0, (2, S))
    _check(kernel, L, tgt, src, X)
