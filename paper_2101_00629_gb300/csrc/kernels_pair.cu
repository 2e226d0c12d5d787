// Pairwise kernel products on CUDA cores: W = Gamma(targets, sources) X.
//
// This is the O(N~^2) step of the IBQ-Galerkin matvec (Sec. 3.1: the rows of
// Gamma are evaluated when needed, never stored) and the kernel product of
// Algorithm 1 in the collocation matvec (Sec. 3.2). Gamma is never stored: every CTA owns 128
// target points (one per thread, coordinates in registers), streams tiles of
// source points and their k vector values through shared memory, evaluates
// the kernel for each (target, source) pair in registers and accumulates
// Gamma_ts * X_s into k per-thread accumulators. FP64 products evaluate the
// kernel in fixed point (pair_fx_kernel); the constant kernel has no
// evaluation and stays in plain FP64 (pair_f64_kernel).
//
// The source range is split across blockIdx.y so that small target counts
// still fill the GPU; each split writes its partial sums to scratch and a
// second kernel adds the splits in a fixed order (deterministic results) and
// applies sigma^2 and the optional per-target scale (J of Sec. 3.1).
#include <cmath>
#include <type_traits>

#include "fixed_gamma.cuh"
#include "kernel_eval.cuh"
#include "kernels_tc.h"
#include "kl_internal.h"

namespace kl {

namespace {

constexpr int kTgt = 128;  // targets per CTA (= threads)
constexpr int kSrc = 128;  // sources per shared-memory tile

template <int KIND, int KB>
__global__ void __launch_bounds__(kTgt) pair_f64_kernel(
    const double* __restrict__ tx, const double* __restrict__ ty, const double* __restrict__ tz,
    int64_t T, const double* __restrict__ sx, const double* __restrict__ sy,
    const double* __restrict__ sz, int64_t S, const double* __restrict__ X, int64_t ldx, int k,
    int c0, double a, double* __restrict__ part, int64_t per_split) {
    chain_wait();
    __shared__ double s_x[kSrc], s_y[kSrc], s_z[kSrc];
    __shared__ double s_v[kSrc][KB];
    const int64_t t = int64_t(blockIdx.x) * kTgt + threadIdx.x;
    const int split = blockIdx.y;
    const int64_t s0 = int64_t(split) * per_split;
    const int64_t s1 = min(S, s0 + per_split);
    const double px = t < T ? tx[t] : 0.0, py = t < T ? ty[t] : 0.0, pz = t < T ? tz[t] : 0.0;
    const int kc = min(KB, k - c0);
    double acc[KB];
#pragma unroll
    for (int c = 0; c < KB; ++c) acc[c] = 0.0;
    for (int64_t base = s0; base < s1; base += kSrc) {
        const int n = int(s1 - base < kSrc ? s1 - base : int64_t(kSrc));
        __syncthreads();
        for (int i = threadIdx.x; i < kSrc; i += kTgt) {
            const bool v = i < n;
            s_x[i] = v ? sx[base + i] : 0.0;
            s_y[i] = v ? sy[base + i] : 0.0;
            s_z[i] = v ? sz[base + i] : 0.0;
        }
        for (int i = threadIdx.x; i < kSrc * KB; i += kTgt) {
            const int c = i / kSrc, j = i - c * kSrc;
            s_v[j][c] = (j < n && c < kc) ? X[base + j + int64_t(c0 + c) * ldx] : 0.0;
        }
        __syncthreads();
        for (int j = 0; j < n; ++j) {
            const double g = gamma64<KIND>(px - s_x[j], py - s_y[j], pz - s_z[j], a);
#pragma unroll
            for (int c = 0; c < KB; ++c) acc[c] = fma(g, s_v[j][c], acc[c]);
        }
    }
    if (t < T) {
        for (int c = 0; c < kc; ++c) part[(int64_t(split) * k + c0 + c) * T + t] = acc[c];
    }
}

// Sources as a tensor grid n[0] x n[1] x n[2] (index i0 + n0 (i1 + n1 i2)) cut
// into blocks of 2^s[0] x 2^s[1] x 2^s[2] points, 32 or fewer.
struct SrcGrid {
    int64_t n[3];
    uint32_t nb[3];
    int s[3];
    __host__ __device__ int64_t groups() const { return int64_t(nb[0]) * nb[1] * nb[2]; }
    // source of a lane of a group, -1 past the edge of the grid
    __device__ int64_t source(uint32_t g, uint32_t lane) const {
        const uint32_t g1 = g / nb[0], b0 = g - g1 * nb[0], b2 = g1 / nb[1], b1 = g1 - b2 * nb[1];
        const int64_t i0 = (int64_t(b0) << s[0]) + (lane & ((1u << s[0]) - 1u));
        const int64_t i1 = (int64_t(b1) << s[1]) + ((lane >> s[0]) & ((1u << s[1]) - 1u));
        const int64_t i2 = (int64_t(b2) << s[2]) + ((lane >> (s[0] + s[1])) & ((1u << s[2]) - 1u));
        const bool in = i0 < n[0] && i1 < n[1] && i2 < n[2] && (lane >> (s[0] + s[1] + s[2])) == 0;
        return in ? i0 + n[0] * (i1 + n[1] * i2) : -1;
    }
};

struct FxScale {
    uint64_t m;  // scale of a distance in base-2 exponents: m 2^e
    int e;
    float f;     // the same, rounded
};

__device__ const fx::Exp2Table g_exp2 = fx::Exp2Table();

// FP64 product with the kernel values in fixed point (fixed_gamma.cuh).
//
// Per pair the FP64 formula costs 20 to 40 FP64 operations for the value and
// k for the product, on a pipe that takes 1.6 per clock and SM. Here the
// value is evaluated in integers and, wherever the kernel varies little over
// a group of 32 sources, the product is too: value and vector entries become
// 57-bit numbers relative to the largest of the group, in two limbs of 28 and
// 29 bits, and three 32 x 32 -> 64-bit multiply-adds per column sum the group
// exactly (the product of the two low limbs lies below the last bit kept).
// One FP64 FMA per column and group adds the group to the running sum.
//
// The integer form is off by at most
//     2^-58 G (W + (n / 2 + c + 1) M),  W = sum |x|,
// in a group with values below G and n non-zero entries below M, c of them
// rounded: truncation of the values (half a unit is added back to each), rounding
// of the entries and of the sum, and the dropped product (half of its range is
// added back). An FP64 evaluation may be off by 2^-53 (0.75 + 0.35 t) g |x| in a
// term (rounding of the exponential and one rounding of its exponent t, 2^-54 t
// ln 2) and by 2^-53 g |x| for each of the r additions that follow, of which half
// is counted. A group takes the integer form where its bound is the smaller one
// in every column. The sum over g v, v = (0.75 + r / 2) |x|, is at least V = sum v
// times the value at the mean squared distance with the weights v (all kernels
// are convex in it; the separable one in each direction), which mean and
// variance of the positions give; 0.35 t g is at least that of the farthest
// source:
//     V g(mean) + 0.35 t_max W g(t_max) >= 2^-5 G (W + (n / 2 + c + 1) M).
// Groups with entries of one size pass up to values of 2^-6 G, groups that a far
// and late entry dominates hardly ever. On lines of 0.25 to 5.5 correlation
// lengths with equal, normal, graded, single and dominating entries the form
// then is as exact as FP64 or better wherever it is taken, rms and largest
// error. A limit on the values alone let through ten times FP64's error (an
// entry of 1 behind 31 below 1e-8: 25 against 2.4 units of 2^-53 of sum g |x|, rms).
//
// A group is a block of the sources' tensor grid (SrcGrid), as near a cube as
// the grid's spacing allows: 32 consecutive points of the half cylinder's
// angle would span a third of it and leave most groups too wide.
//
// Each lane bounds the exponents of its targets against the box of the
// group's source points, and the warp takes the first path that all its lanes
// allow:
//   products in integers   exponents close to each other, as above
//   products in FP64       exponents in the fixed-point range
//   all in FP64            anything else: points too far apart for the range
//                          (exponents above 120 to 1000), infinities, NaN,
//                          entries below 2^-322
//
// Measured against the FP64 formula for every pair: 5003 x 20011 scattered
// points, Matern-3/2, 3 columns, 8.14 -> 0.86 ms; half-cylinder Galerkin
// operator, Euclidean exponential, 8 columns, 1.5e8 pairs, 10.7 -> 1.72 ms, and
// its degree-6 Gaussian collocation operator, 3.7e8 pairs, 20.3 -> 3.65 ms (every
// group on FP64 products: 5 ms, that pipe 93 % busy; deciding without the
// entries took 0.84, 1.60 and 2.94 ms at the errors above). Bound by the integer
// pipes: 83 to 172 instructions per pair and about seven per column, three of
// them 32 x 32 -> 64-bit multiply-adds of four issue cycles. Two targets per
// thread were 5 to 20 % slower (registers). Half of a group's columns per warp
// with 16 columns: 16^3 cube, Gaussian collocation, 8.9 -> 8.0 ms (7.6 ms without
// the rule on the entries).
template <int KIND, int KB>
__global__ void __launch_bounds__(kTgt, KB > 8 ? 3 : 5) pair_fx_kernel(
    const double* __restrict__ tx, const double* __restrict__ ty, const double* __restrict__ tz,
    int64_t T, const double* __restrict__ sx, const double* __restrict__ sy,
    const double* __restrict__ sz, SrcGrid sg, const double* __restrict__ X, int64_t ldx, int k,
    int c0, double a, FxScale sc, double* __restrict__ part, int64_t per_split) {
    chain_wait();
    constexpr int NG = KB > 8 ? 2 : 4;  // groups per stage
    constexpr int ST = 32 * NG;
    // each warp stages a group's columns, two warps half of them each with two
    // groups per stage
    constexpr int PARTS = kTgt / 32 / NG, KP = KB / PARTS;
    static_assert(PARTS * NG * 32 == kTgt && KP * PARTS == KB, "all warps stage");
    constexpr int Q = fx::Format<KIND>::kCoord, QA = fx::Format<KIND>::kArg;
    __shared__ __align__(16) uint64_t s_tab[2048];
    __shared__ __align__(16) uint64_t s_c[ST][4];
    __shared__ __align__(16) int2 s_xl[ST][KB];
    __shared__ __align__(16) double s_xd[ST][KB];
    __shared__ float s_box[NG][6], s_quick[NG][PARTS];
    __shared__ float4 s_mean[NG][KB], s_var[NG][KB];
    __shared__ int s_emax[NG][KB];
    __shared__ int64_t s_mean_low[NG][KB];
    __shared__ int s_special[NG][PARTS], s_count[NG], s_emin[NG][PARTS];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    for (int i = tid; i < 1024; i += kTgt)
        reinterpret_cast<ulonglong2*>(s_tab)[i] = reinterpret_cast<const ulonglong2*>(g_exp2.v)[i];
    const int split = blockIdx.y;
    // groups [s0, s1) of this split
    const int64_t s0 = int64_t(split) * per_split;
    const int64_t s1 = min(sg.groups(), s0 + per_split);
    const int64_t t0 = int64_t(blockIdx.x) * kTgt;
    const int kc = min(KB, k - c0);
    // boxes are taken relative to the block's first target
    const double rx = tx[t0], ry = ty[t0], rz = tz[t0];
    const int64_t tc = min(t0 + tid, T - 1);
    const double px = tx[tc], py = ty[tc], pz = tz[tc];
    const uint64_t ux = fx::to_fixed<Q>(px, sc.m, sc.e), uy = fx::to_fixed<Q>(py, sc.m, sc.e),
                   uz = fx::to_fixed<Q>(pz, sc.m, sc.e);
    const float p[3] = {float(px - rx) * sc.f, float(py - ry) * sc.f, float(pz - rz) * sc.f};
    const bool tfinite = isfinite(p[0]) && isfinite(p[1]) && isfinite(p[2]);
    double acc[KB];
#pragma unroll
    for (int c = 0; c < KB; ++c) acc[c] = 0.0;
    for (int64_t base = s0; base < s1; base += NG) {
        const int ng = int(s1 - base < NG ? s1 - base : int64_t(NG));
        __syncthreads();
        // one warp per group (or half of its columns), one source per lane; a block of the grid that
        // reaches over its edge leaves lanes without a source, the others
        // move together
        if (const int g = warp / PARTS, share = warp % PARTS; g < ng) {
            const int64_t sj = sg.source(uint32_t(base) + g, lane);
            const unsigned have = __ballot_sync(0xffffffffu, sj >= 0);
            const bool v = sj >= 0;
            const int j = g * 32 + __popc(have & ((1u << lane) - 1u));
            const int64_t sl = __shfl_sync(0xffffffffu, (long long)sj, __ffs(int(have)) - 1);
            const int64_t sv = v ? sj : sl;
            const double x = sx[sv], y = sy[sv], z = sz[sv];
            if (v && share == 0) {
                s_c[j][0] = fx::to_fixed<Q>(x, sc.m, sc.e);
                s_c[j][1] = fx::to_fixed<Q>(y, sc.m, sc.e);
                s_c[j][2] = fx::to_fixed<Q>(z, sc.m, sc.e);
                s_c[j][3] = uint64_t(sj);
            }
            float lo[3] = {float(x - rx) * sc.f, float(y - ry) * sc.f, float(z - rz) * sc.f}, hi[3];
            bool bad = !(isfinite(lo[0]) && isfinite(lo[1]) && isfinite(lo[2]));
            int emin = 2047;
            const float rel[3] = {lo[0], lo[1], lo[2]};
            float quick = 16384.0f;
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                hi[q] = lo[q];
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    lo[q] = fminf(lo[q], __shfl_xor_sync(0xffffffffu, lo[q], o));
                    hi[q] = fmaxf(hi[q], __shfl_xor_sync(0xffffffffu, hi[q], o));
                }
            }
#pragma unroll
            for (int cc = 0; cc < KP; ++cc) {
                const int c = share * KP + cc;
                const double xv = (v && c < kc) ? X[sj + int64_t(c0 + c) * ldx] : 0.0;
                if (v) s_xd[j][c] = xv;
                const uint64_t b = uint64_t(__double_as_longlong(xv)) & 0x7fffffffffffffffull;
                const int ef = int(b >> 52);
                const int e = ef ? ef : (b ? 1 : 0);
                int emax = __reduce_max_sync(0xffffffffu, e);
                bad = bad || emax == 2047 || (emax > 0 && emax < 700);
                if (emax == 0) emax = 1079;
                emin = min(emin, emax);
                // |x| 2^(1078 - emax), rounded: at most 2^56
                const uint64_t m = ((b & 0xfffffffffffffull) | (ef ? uint64_t(1) << 52 : 0)) << 3;
                const int rs = emax - e;
                int64_t xi = 0;
                if (rs <= 57) xi = int64_t((m + (rs ? uint64_t(1) << (rs - 1) : 0)) >> rs);
                if (xv < 0.0) xi = -xi;
                const int32_t x1 = int32_t((xi + (1 << 27)) >> 28);
                // entries' sizes (2^26 at most), their sum, and that of the
                // weights v of the rule above; a mean position out of reach
                // until it is formed below
                const unsigned some = __ballot_sync(0xffffffffu, b != 0);
                const int cut = __popc(__ballot_sync(0xffffffffu, rs > 3 && b != 0));
                const unsigned size = unsigned(x1 < 0 ? -x1 : x1) >> 2;
                const float sum = float(__reduce_add_sync(0xffffffffu, size));
                // 4 v 2^-16, at most 65 * 2^10 (30 bits with the positions)
                const int weight = int(size >> 16) * int(2 * __popc(some >> lane) + 1);
                const float total = float(__reduce_add_sync(0xffffffffu, weight));
                const float d = 32.0f / (sum + float(__popc(some) + 2 * cut + 2) * 33554432.0f);
                if (some) quick = fminf(quick, 16384.0f * total * d);
                if (lane == 0) {
                    s_mean[g][c] = make_float4(1e18f, 1e18f, 1e18f, some ? 16384.0f * total * d : 0.0f);
                    s_var[g][c] = make_float4(0.0f, 0.0f, 0.0f, some ? 0.35f * sum * d : 1e30f);
                }
                const int32_t x0 = int32_t(xi - (int64_t(x1) << 28));
                if (v) s_xl[j][c] = make_int2(x1, x0);
                const int half = __reduce_add_sync(0xffffffffu, (x1 + x0) >> 3);
                if (lane == 0) {
                    s_emax[g][c] = emax;
                    s_mean_low[g][c] = int64_t(half) * 4 + (1 << 27);
                }
            }
            // the mean positions, where the quick test may fail: elsewhere the
            // exponents of the box lie within its diameter of each other (not
            // the Gaussian's, which grow with the distance)
            const float diameter = (hi[0] - lo[0]) + (hi[1] - lo[1]) + (hi[2] - lo[2]);
            if (KIND == KL_KERNEL_GAUSS || !(quick * ex2_approx(-1.01f * diameter - 1.1f) >= 1.0f)) {
                // positions in the box, 500 units to its largest half edge, and
                // their squares (EXP_SEP: one by one) over 2048
                const float half_edge = 0.5f * fmaxf(hi[0] - lo[0], fmaxf(hi[1] - lo[1], hi[2] - lo[2]));
                const float unit = half_edge * 0.002f, per_unit = half_edge > 0.0f ? 500.0f / half_edge : 0.0f;
                float centre[3];
                int at[3], sq[3];
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    centre[q] = 0.5f * (lo[q] + hi[q]);
                    at[q] = __float2int_rn((rel[q] - centre[q]) * per_unit);
                    sq[q] = at[q] * at[q];
                }
                if (KIND != KL_KERNEL_EXP_SEP) sq[0] += sq[1] + sq[2];
#pragma unroll
                for (int q = 0; q < 3; ++q) sq[q] = (sq[q] + 1024) >> 11;
#pragma unroll
                for (int cc = 0; cc < KP; ++cc) {
                    const int c = share * KP + cc;
                    const int x1 = v ? s_xl[j][c].x : 0;
                    const unsigned some = __ballot_sync(0xffffffffu, v && s_xd[j][c] != 0.0);
                    const int weight = int(unsigned(x1 < 0 ? -x1 : x1) >> 18) * int(2 * __popc(some >> lane) + 1);
                    const float r = 1.0f / float(__reduce_add_sync(0xffffffffu, weight));
                    const float y0 = float(__reduce_add_sync(0xffffffffu, weight * at[0])) * r;
                    const float y1 = float(__reduce_add_sync(0xffffffffu, weight * at[1])) * r;
                    const float y2 = float(__reduce_add_sync(0xffffffffu, weight * at[2])) * r;
                    const float q0 = 2048.0f * float(__reduce_add_sync(0xffffffffu, weight * sq[0])) * r;
                    float v0 = q0 - y0 * y0, v1 = 0.0f, v2 = 0.0f;
                    if (KIND == KL_KERNEL_EXP_SEP) {
                        v1 = 2048.0f * float(__reduce_add_sync(0xffffffffu, weight * sq[1])) * r - y1 * y1;
                        v2 = 2048.0f * float(__reduce_add_sync(0xffffffffu, weight * sq[2])) * r - y2 * y2;
                    } else {
                        v0 -= y1 * y1 + y2 * y2;
                    }
                    if (lane == 0 && some) {
                        s_mean[g][c].x = fmaf(y0, unit, centre[0]);
                        s_mean[g][c].y = fmaf(y1, unit, centre[1]);
                        s_mean[g][c].z = fmaf(y2, unit, centre[2]);
                        s_var[g][c].x = fmaxf(v0, 0.0f) * (unit * unit);
                        s_var[g][c].y = fmaxf(v1, 0.0f) * (unit * unit);
                        s_var[g][c].z = fmaxf(v2, 0.0f) * (unit * unit);
                    }
                }
            }
            const bool any_bad = __any_sync(0xffffffffu, bad);
            if (lane == 0) {
                s_special[g][share] = any_bad;
                s_emin[g][share] = emin;
                s_quick[g][share] = quick;
                if (share == 0) {
                    s_count[g] = __popc(have);
#pragma unroll
                    for (int q = 0; q < 3; ++q) s_box[g][q] = lo[q], s_box[g][3 + q] = hi[q];
                }
            }
        }
        __syncthreads();
        for (int g = 0; g < ng; ++g) {
            const int j0 = g * 32, j1 = j0 + s_count[g];
            // bounds of the exponents over the box; the slack covers the
            // rounding of the single-precision coordinates
            float tlo = 0.0f, thi = 0.0f;
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const float lo = s_box[g][q], hi = s_box[g][3 + q];
                const float eps = 1e-6f * (fabsf(lo) + fabsf(hi) + fabsf(p[q]));
                const float dl = fmaxf(fmaxf(lo - p[q], p[q] - hi) - eps, 0.0f);
                const float dh = fmaxf(p[q] - lo, hi - p[q]) + eps;
                tlo += KIND == KL_KERNEL_EXP_SEP ? dl : dl * dl;
                thi += KIND == KL_KERNEL_EXP_SEP ? dh : dh * dh;
            }
            if (KIND == KL_KERNEL_EXP || KIND == KL_KERNEL_MATERN32) {
                tlo = sqrtf(tlo);
                thi = sqrtf(thi);
            }
            const bool in_range = tfinite && !(s_special[g][0] | s_special[g][PARTS - 1]) && thi < fx::Format<KIND>::kMaxArg;
            const float far = thi + 1e-9f;
            int gm = 0;
            if (KIND == KL_KERNEL_MATERN32) {
                const float fh = 1.0f + 0.6931472f * thi;
                gm = 1 + int(log2f(fh) + 1e-3f);  // 1 + t ln 2 < 2^gm
                tlo -= log2f(1.0f + 0.6931472f * tlo);
                thi -= log2f(fh);
            }
            tlo = fmaxf(tlo * (1.0f - 1e-5f) - 1e-3f, 0.0f);
            thi = thi * (1.0f + 1e-5f) + 1e-3f;
            const int n0 = int(fminf(tlo, 1000.0f));
            // the group's scale 2^(emax - 56 - n0) is a normal number in every
            // column (far Gaussian groups: n0 reaches 999)
            bool narrow = thi - float(n0) < 14.0f && n0 <= min(s_emin[g][0], s_emin[g][PARTS - 1]) - 57;
            const float farthest = ex2_approx(float(n0) - thi);
            // the rule with the farthest value in place of the mean, then the
            // rule itself
            if (!__all_sync(0xffffffffu, in_range && narrow && fminf(s_quick[g][0], s_quick[g][PARTS - 1]) * farthest >= 1.0f)) {
#pragma unroll
                for (int c = 0; c < KB; ++c) {
                    const float4 mean = s_mean[g][c], var = s_var[g][c];
                    const float dx = p[0] - mean.x, dy = p[1] - mean.y, dz = p[2] - mean.z;
                    float t, f = 1.0f;
                    if (KIND == KL_KERNEL_EXP_SEP)
                        t = sqrt_approx(fmaf(dx, dx, var.x)) + sqrt_approx(fmaf(dy, dy, var.y)) + sqrt_approx(fmaf(dz, dz, var.z));
                    else
                        t = fmaf(dx, dx, fmaf(dy, dy, fmaf(dz, dz, var.x)));
                    if (KIND == KL_KERNEL_EXP || KIND == KL_KERNEL_MATERN32) t = sqrt_approx(t);
                    if (KIND == KL_KERNEL_MATERN32) f = 1.0f + 0.6931472f * t;
                    t = fmaf(t, 1.0f + 1e-5f, 1e-3f);
                    narrow = narrow && fmaf(mean.w * f, ex2_approx(float(n0) - t), var.w * (far * farthest)) >= 1.0f;
                }
            }
            if (__all_sync(0xffffffffu, in_range && narrow)) {
                int64_t hi[KB], mid[KB];
#pragma unroll
                for (int c = 0; c < KB; ++c) hi[c] = 0, mid[c] = 0;
#pragma unroll 2
                for (int j = j0; j < j1; ++j) {
                    const ulonglong2 qxy = *reinterpret_cast<const ulonglong2*>(s_c[j]);
                    const uint64_t t = fx::exponent<KIND>(fx::absdiff(ux, qxy.x), fx::absdiff(uy, qxy.y),
                                                          fx::absdiff(uz, s_c[j][2]));
                    uint32_t nt, g1, g0;
                    uint64_t E = fx::exp2_neg<QA>(t, s_tab, nt);
                    if (KIND == KL_KERNEL_MATERN32) {
                        E = fx::mulhi64(E, fx::matern_factor(t) << (9 - gm)) >> (6 + int(nt) - n0 - gm);
                        g1 = uint32_t(E >> 28);
                        g0 = uint32_t(E) & 0xfffffffu;
                    } else {
                        const uint32_t s = 2u + nt - uint32_t(n0);
                        g1 = uint32_t(E >> 32) >> s;
                        g0 = __funnelshift_r(uint32_t(E), uint32_t(E >> 32), s) >> 4;
                    }
#pragma unroll
                    for (int c = 0; c < KB; ++c) {
                        int2 xl;  // two columns per 16-byte load
                        if (KB == 1) {
                            xl = s_xl[j][c];
                        } else {
                            const int4 x2 = *reinterpret_cast<const int4*>(&s_xl[j][c & ~1]);
                            xl = c & 1 ? make_int2(x2.z, x2.w) : make_int2(x2.x, x2.y);
                        }
                        hi[c] = fx::madwide_s(int32_t(g1), xl.x, hi[c]);
                        mid[c] = fx::madwide_s(int32_t(g1), xl.y, mid[c]);
                        mid[c] = fx::madwide_s(int32_t(g0), xl.x, mid[c]);
                    }
                }
#pragma unroll
                for (int c = 0; c < KB; ++c) {
                    const int64_t sum = hi[c] + ((mid[c] + s_mean_low[g][c]) >> 28);
                    const double f = __longlong_as_double((long long)(s_emax[g][c] - 56 - n0) << 52);
                    acc[c] = fma(double(sum), f, acc[c]);
                }
            } else if (__all_sync(0xffffffffu, in_range)) {
                // the group's own sum first, as in the integer form: one
                // rounding at the size of the running sum, not 32
                double sum[KB];
#pragma unroll
                for (int c = 0; c < KB; ++c) sum[c] = 0.0;
                for (int j = j0; j < j1; ++j) {
                    const uint64_t t = fx::exponent<KIND>(fx::absdiff(ux, s_c[j][0]), fx::absdiff(uy, s_c[j][1]),
                                                          fx::absdiff(uz, s_c[j][2]));
                    uint32_t nt;
                    const uint64_t E = fx::exp2_neg<QA>(t, s_tab, nt);
                    double gv = fx::to_double(E, nt);
                    if (KIND == KL_KERNEL_MATERN32) gv *= double(fx::matern_factor(t)) * 2.7755575615628914e-17;  // 2^-55
#pragma unroll
                    for (int c = 0; c < KB; ++c) sum[c] = fma(gv, s_xd[j][c], sum[c]);
                }
#pragma unroll
                for (int c = 0; c < KB; ++c) acc[c] += sum[c];
            } else {
                for (int j = j0; j < j1; ++j) {
                    const int64_t sj = int64_t(s_c[j][3]);
                    const double gv = gamma64<KIND>(px - sx[sj], py - sy[sj], pz - sz[sj], a);
#pragma unroll
                    for (int c = 0; c < KB; ++c) acc[c] = fma(gv, s_xd[j][c], acc[c]);
                }
            }
        }
    }
    if (t0 + tid < T) {
#pragma unroll
        for (int c = 0; c < KB; ++c)
            if (c < kc) part[(int64_t(split) * k + c0 + c) * T + t0 + tid] = acc[c];
    }
}

// FP32 product: R targets per thread, so that a source's coordinates (one
// 16-byte load) and its KB entries serve R pairs. Bound by instruction issue:
// about 12 per value (two of them special-function), KB per product, and by
// the FP64 additions of the tile sums. 2688 x 82368 points, Matern-3/2, whole
// application: 5 columns 245 -> 205 us (198 us with dependent launches), 16
// columns 455 -> 410 us against one target per thread, scalar coordinate loads
// and 8 columns at least.
template <int KIND, int KB, int R>
__global__ void __launch_bounds__(kTgt) pair_f32_kernel(
    const float* __restrict__ tx, const float* __restrict__ ty, const float* __restrict__ tz,
    int64_t T, const float* __restrict__ sx, const float* __restrict__ sy,
    const float* __restrict__ sz, int64_t S, const double* __restrict__ X, int64_t ldx, int k,
    int c0, float a, float a2, double* __restrict__ part, int64_t per_split) {
    chain_wait();
    __shared__ float4 s_c[kSrc];
    __shared__ __align__(16) float s_v[kSrc][KB];
    const int64_t t0 = int64_t(blockIdx.x) * (kTgt * R) + threadIdx.x;
    const int split = blockIdx.y;
    const int64_t s0 = int64_t(split) * per_split;
    const int64_t s1 = min(S, s0 + per_split);
    float px[R], py[R], pz[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int64_t t = t0 + r * kTgt;
        px[r] = t < T ? tx[t] : 0.f, py[r] = t < T ? ty[t] : 0.f, pz[r] = t < T ? tz[t] : 0.f;
    }
    const int kc = min(KB, k - c0);
    float acc[R][KB];
    double accd[R][KB];
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int c = 0; c < KB; ++c) acc[r][c] = 0.f, accd[r][c] = 0.0;
    for (int64_t base = s0; base < s1; base += kSrc) {
        const int n = int(s1 - base < kSrc ? s1 - base : int64_t(kSrc));
        __syncthreads();
        for (int i = threadIdx.x; i < kSrc; i += kTgt) {
            const bool v = i < n;
            s_c[i] = v ? make_float4(sx[base + i], sy[base + i], sz[base + i], 0.f) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        for (int i = threadIdx.x; i < kSrc * KB; i += kTgt) {
            const int c = i / kSrc, j = i - c * kSrc;
            s_v[j][c] = (j < n && c < kc) ? float(X[base + j + int64_t(c0 + c) * ldx]) : 0.f;
        }
        __syncthreads();
#pragma unroll 2
        for (int j = 0; j < n; ++j) {
            const float4 q = s_c[j];
            float g[R];
#pragma unroll
            for (int r = 0; r < R; ++r) g[r] = gamma32<KIND>(px[r] - q.x, py[r] - q.y, pz[r] - q.z, a, a2);
#pragma unroll
            for (int c = 0; c < KB; ++c) {
                const float v = s_v[j][c];
#pragma unroll
                for (int r = 0; r < R; ++r) acc[r][c] = fmaf(g[r], v, acc[r][c]);
            }
        }
        // flush the FP32 tile sums into FP64 once per tile
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
            for (int c = 0; c < KB; ++c) accd[r][c] += double(acc[r][c]), acc[r][c] = 0.f;
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int64_t t = t0 + r * kTgt;
        if (t < T) {
#pragma unroll
            for (int c = 0; c < KB; ++c)
                if (c < kc) part[(int64_t(split) * k + c0 + c) * T + t] = accd[r][c];
        }
    }
}

// Y = sigma^2 post .* (sum of the splits' partial sums). A block serves 32
// points of one column, warp y the y-th eighth of the splits; warp 0 adds the
// eight in order. With one thread per output, 64 loads one after the other
// took 15 to 20 us (cold) for a few thousand points.
constexpr int kRedSlices = 8;
__global__ void __launch_bounds__(32 * kRedSlices) pair_reduce_kernel(const double* __restrict__ part, int splits,
                                                                      int64_t T, int k, double sigma2,
                                                                      const double* __restrict__ post, double* Y,
                                                                      int64_t ldy) {
    chain_wait();
    __shared__ double sh[kRedSlices][32];
    const int lane = threadIdx.x & 31, sl = threadIdx.x >> 5;
    const int per = (splits + kRedSlices - 1) / kRedSlices;
    const int sp0 = min(splits, sl * per), sp1 = min(splits, sp0 + per);
    const int64_t tiles = (T + 31) / 32;
    for (int64_t b = blockIdx.x; b < tiles * k; b += gridDim.x) {
        const int64_t c = b / tiles, t = (b - c * tiles) * 32 + lane;
        double s = 0.0;
        if (t < T) {
            const double* p = part + c * T + t;
            const int64_t step = int64_t(k) * T;
#pragma unroll 8
            for (int sp = sp0; sp < sp1; ++sp) s += p[sp * step];
        }
        __syncthreads();
        sh[sl][lane] = s;
        __syncthreads();
        if (sl == 0 && t < T) {
#pragma unroll
            for (int q = 1; q < kRedSlices; ++q) s += sh[q][lane];
            s *= sigma2;
            if (post) s *= post[t];
            Y[c * ldy + t] = s;
        }
    }
}

cudaError_t run_pair_reduce(const double* part, int splits, int64_t T, int k, double sigma2, const double* post,
                            double* Y, int64_t ldy, cudaStream_t s) {
    const int64_t blocks = (T + 31) / 32 * k;
    const int g = int(std::min<int64_t>(blocks, int64_t(device_sm_count()) * 32));
    launch_chain(pair_reduce_kernel, g < 1 ? 1 : g, 32 * kRedSlices, 0, s, part, splits, T, k, sigma2, post, Y, ldy);
    return cudaGetLastError();
}

// Scale of a distance (Gauss: its square root is taken) in base-2 exponents,
// to 64 bits: a log2(e) or sqrt(a log2(e)).
// 1 / L or 1 / L^2 beyond the FP64 range (L below 1e-154 for the Gaussian)
// leaves no scale: infinite, so that every group takes the FP64 formula.
FxScale fx_scale(int kind, double a) {
    if (!std::isfinite(a)) return {0, 0, INFINITY};
    int e;
    const double f = std::frexp(a, &e);                           // a = f 2^e, f in [1/2, 1)
    const uint64_t m = uint64_t(std::ldexp(f, 53));               // exact
    unsigned __int128 p = (unsigned __int128)m * 0xb8aa3b295c17f0bcull;  // log2(e) 2^63; p in [2^115, 2^117)
    e -= 53 + 63;                                                 // a log2(e) = p 2^e
    FxScale sc;
    if (kind == KL_KERNEL_GAUSS) {
        // p 2^10 or 2^11 (even exponent) has 125 to 128 bits: its root 63 or 64
        const int s = (e & 1) ? 11 : 10;
        p <<= s;
        e -= s;
        unsigned __int128 r = 0;
        for (int b = 63; b >= 0; --b) {
            const unsigned __int128 q = r | ((unsigned __int128)1 << b);
            if (q * q <= p) r = q;
        }
        sc.m = uint64_t(r);
        sc.e = e / 2;
    } else {
        sc.m = uint64_t(p >> 53);
        sc.e = e + 53;
    }
    sc.f = float(std::ldexp(double(sc.m), sc.e));
    return sc;
}

template <int KIND>
void launch_f64(const PairArgs& a, int c0, int64_t per_split, cudaStream_t s) {
    const dim3 grid(unsigned((a.T + kTgt - 1) / kTgt), unsigned(a.splits));
    const int kc = a.k - c0;
    if (kc <= 8)
        launch_kernel(few_blocks(grid), pair_f64_kernel<KIND, 8>, grid, kTgt, 0, s, a.tx, a.ty, a.tz, a.T, a.sx, a.sy, a.sz, a.S, a.X, a.ldx, a.k, c0, a.ks.a, a.scratch, per_split);
    else if (kc <= 16)
        launch_kernel(few_blocks(grid), pair_f64_kernel<KIND, 16>, grid, kTgt, 0, s, a.tx, a.ty, a.tz, a.T, a.sx, a.sy, a.sz, a.S, a.X, a.ldx, a.k, c0, a.ks.a, a.scratch, per_split);
    else
        launch_kernel(few_blocks(grid), pair_f64_kernel<KIND, 32>, grid, kTgt, 0, s, a.tx, a.ty, a.tz, a.T, a.sx, a.sy, a.sz, a.S, a.X, a.ldx, a.k, c0, a.ks.a, a.scratch, per_split);
}

// Blocks of the source grid: from one point, double the block along the
// direction in which it is shortest until it has 32; fewer (down to 4) where
// the splits would outnumber the blocks.
SrcGrid src_grid(const PairArgs& a) {
    SrcGrid g{};
    for (int bits = 5; bits >= 2; --bits) {
        double h[3];
        for (int d = 0; d < 3; ++d) {
            g.n[d] = a.sn[0] > 0 ? a.sn[d] : (d == 0 ? a.S : 1);
            h[d] = a.sn[0] > 0 ? a.sh[d] : 1.0;
            g.s[d] = 0;
        }
        for (int left = bits; left > 0; --left) {
            int best = -1;
            for (int d = 0; d < 3; ++d)
                if ((int64_t(1) << g.s[d]) < g.n[d] && (best < 0 || h[d] < h[best])) best = d;
            if (best < 0) break;
            ++g.s[best];
            h[best] *= 2.0;
        }
        for (int d = 0; d < 3; ++d) g.nb[d] = uint32_t((g.n[d] + (int64_t(1) << g.s[d]) - 1) >> g.s[d]);
        if (g.groups() >= a.splits) break;
    }
    return g;
}

template <int KIND>
void launch_fx(const PairArgs& a, int c0, const FxScale& sc, const SrcGrid& sg, cudaStream_t s) {
    const int kc = a.k - c0;
    const int64_t per_split = (sg.groups() + a.splits - 1) / a.splits;
    const dim3 grid(unsigned((a.T + kTgt - 1) / kTgt), unsigned(a.splits));
    auto go = [&](auto kb) {
        launch_kernel(few_blocks(grid), pair_fx_kernel<KIND, decltype(kb)::value>, grid, kTgt, 0, s, a.tx, a.ty, a.tz, a.T, a.sx, a.sy, a.sz, sg, a.X, a.ldx, a.k, c0, a.ks.a, sc, a.scratch, per_split);
    };
    if (kc <= 1) go(std::integral_constant<int, 1>{});
    else if (kc <= 2) go(std::integral_constant<int, 2>{});
    else if (kc <= 4) go(std::integral_constant<int, 4>{});
    else if (kc <= 8) go(std::integral_constant<int, 8>{});
    else go(std::integral_constant<int, 16>{});
}

template <int KIND>
cudaError_t launch_kind(const PairArgs& a, bool fp32, cudaStream_t s) {
    const int64_t per_split = (a.S + a.splits - 1) / a.splits;
    if (fp32) {
        KL_RANGE(a.tx32, a.T, float, "pair targets x");
        KL_RANGE(a.ty32, a.T, float, "pair targets y");
        KL_RANGE(a.tz32, a.T, float, "pair targets z");
        KL_RANGE(a.sx32, a.S, float, "pair sources x");
        KL_RANGE(a.sy32, a.S, float, "pair sources y");
        KL_RANGE(a.sz32, a.S, float, "pair sources z");
    } else {
        KL_RANGE(a.tx, a.T, double, "pair targets x");
        KL_RANGE(a.ty, a.T, double, "pair targets y");
        KL_RANGE(a.tz, a.T, double, "pair targets z");
        KL_RANGE(a.sx, a.S, double, "pair sources x");
        KL_RANGE(a.sy, a.S, double, "pair sources y");
        KL_RANGE(a.sz, a.S, double, "pair sources z");
    }
    KL_RANGE(a.X, block_extent(a.S, a.k, a.ldx), double, "pair X");
    KL_RANGE(a.scratch, pair_scratch_doubles(a.T, a.k, a.splits), double, "pair partial sums");
    KL_RANGE(a.Y, block_extent(a.T, a.k, a.ldy), double, "pair Y");
    KL_RANGE(a.post, a.T, double, "pair post");
    const double l2e = 1.4426950408889634074;
    const FxScale sc = fx_scale(KIND, a.ks.a);
    const SrcGrid sg = src_grid(a);
    // columns per pass over the pairs: 32, in fixed point 16 (two 64-bit
    // sums per column in registers)
    const int step = fp32 || KIND == KL_KERNEL_CONST ? 32 : 16;
    for (int c0 = 0; c0 < a.k; c0 += step) {
        const int kc = a.k - c0;
        if (fp32) {
            const float fa = float(a.ks.a), fa2 = float(a.ks.a * l2e);
            auto go = [&](auto kb, auto r) {
                constexpr int KB = decltype(kb)::value, R = decltype(r)::value;
                const dim3 grid(unsigned((a.T + kTgt * R - 1) / (kTgt * R)), unsigned(a.splits));
                launch_kernel(few_blocks(grid), pair_f32_kernel<KIND, KB, R>, grid, kTgt, 0, s, a.tx32, a.ty32, a.tz32, a.T, a.sx32, a.sy32, a.sz32, a.S, a.X, a.ldx, a.k, c0, fa, fa2, a.scratch, per_split);
            };
            using I1 = std::integral_constant<int, 1>;
            using I2 = std::integral_constant<int, 2>;
            if (kc <= 4) go(std::integral_constant<int, 4>{}, I2{});
            else if (kc <= 6) go(std::integral_constant<int, 6>{}, I2{});
            else if (kc <= 8) go(std::integral_constant<int, 8>{}, I2{});
            else if (kc <= 16) go(std::integral_constant<int, 16>{}, I2{});
            else go(std::integral_constant<int, 32>{}, I1{});
        } else {
            if constexpr (KIND == KL_KERNEL_CONST) {
                launch_f64<KIND>(a, c0, per_split, s);
            } else {
                launch_fx<KIND>(a, c0, sc, sg, s);
            }
        }
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return run_pair_reduce(a.scratch, a.splits, a.T, a.k, a.ks.sigma2, a.post, a.Y, a.ldy, s);
}

}  // namespace

int64_t pair_scratch_doubles(int64_t T, int k, int splits) { return T * int64_t(k) * splits; }

int pair_choose_splits(int64_t T, int64_t S, int sm_count, bool fine) {
    // 16 blocks per SM while a split keeps 512 sources. `fine`: 256, and few
    // sources are cut down to 4 per split for one wave of five blocks per SM
    // (216 targets and sources, one column, FP64: 250 us in one split per tile
    // of targets, 12 us in 13, 10 us in 54); the partial sums take more memory,
    // which handles that use this product for a refinement only do without.
    const int64_t tb = (T + kTgt - 1) / kTgt;
    const int64_t many = std::min<int64_t>((16LL * sm_count + tb - 1) / tb, S / (fine ? 256 : 512));
    int64_t few = fine ? std::min<int64_t>(5LL * sm_count / tb, S / 4) : 1;
    // up to 1024 targets: partial sums of eight columns within 1 MiB, which is
    // cheaper to allocate than more
    const int64_t in_mib = (int64_t(1) << 17) / (8 * T);
    if (in_mib >= 16) few = std::min(few, in_mib);
    return int(std::min<int64_t>(64, std::max<int64_t>(1, std::max(many, few))));
}

cudaError_t launch_pair_simt(const PairArgs& a, bool fp32, cudaStream_t s) {
    switch (a.ks.kind) {
        case KL_KERNEL_GAUSS: return launch_kind<KL_KERNEL_GAUSS>(a, fp32, s);
        case KL_KERNEL_EXP_SEP: return launch_kind<KL_KERNEL_EXP_SEP>(a, fp32, s);
        case KL_KERNEL_EXP: return launch_kind<KL_KERNEL_EXP>(a, fp32, s);
        case KL_KERNEL_MATERN32: return launch_kind<KL_KERNEL_MATERN32>(a, fp32, s);
        default: return launch_kind<KL_KERNEL_CONST>(a, fp32, s);
    }
}

}  // namespace kl
