// Diagnostics reduction: energy (Eq. 27), div B statistics and a non-finite
// count in one pass over the state, reduced in FP64 with Neumaier-compensated
// sums in a fixed order (the result depends only on the lattice size, not on
// scheduling).
//
// Pass 1 (diag_partial): block b takes rows b, b + G, b + 2G, ...; every
// thread keeps compensated sums of its per-row sums; the block combines its
// threads in a fixed tree and writes one partial record to scratch.
// Pass 2 (diag_final): one block combines the G partials in a fixed tree.
#include <math.h>

#include "qla_internal.h"

namespace qla {

namespace {

constexpr int DIAG_THREADS = 256;

struct CSum {
    double s, c;
    __device__ __forceinline__ void add(double v) {
        const double t = s + v;
        if (fabs(s) >= fabs(v)) c += (s - t) + v;
        else c += (v - t) + s;
        s = t;
    }
    __device__ __forceinline__ void merge(const CSum &o) {
        add(o.s);
        c += o.c;
    }
};

struct Partial {
    double e_s, e_c, d_s, d_c, dmax, bmax;
    unsigned long long nonfinite;
    unsigned long long pad;
};

template <typename T>
__device__ __forceinline__ bool finite_val(T v) {
    return isfinite(v);
}

__device__ __forceinline__ void merge_into(Partial &a, const Partial &b) {
    CSum es{a.e_s, a.e_c}, ds{a.d_s, a.d_c};
    es.merge(CSum{b.e_s, b.e_c});
    ds.merge(CSum{b.d_s, b.d_c});
    a.e_s = es.s; a.e_c = es.c; a.d_s = ds.s; a.d_c = ds.c;
    a.dmax = fmax(a.dmax, b.dmax);
    a.bmax = fmax(a.bmax, b.bmax);
    a.nonfinite += b.nonfinite;
}

// The block's threads combined in a fixed tree; thread 0 writes the record.
__device__ __forceinline__ void block_reduce_write(const Partial &mine, Partial *__restrict__ part) {
    __shared__ Partial sh[DIAG_THREADS];
    sh[threadIdx.x] = mine;
    __syncthreads();
    for (int w = DIAG_THREADS / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) {
            Partial a = sh[threadIdx.x];
            merge_into(a, sh[threadIdx.x + w]);
            sh[threadIdx.x] = a;
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = sh[0];
}

template <typename T>
__global__ void __launch_bounds__(DIAG_THREADS) diag_partial(const T *__restrict__ q, int Nx, int Ny,
                                                             Partial *__restrict__ part) {
    const size_t P = size_t(Nx) * size_t(Ny);
    const T *q3 = q + 3 * P, *q4 = q + 4 * P;
    CSum e{0.0, 0.0}, d{0.0, 0.0};
    double dmax = 0.0, b2max = 0.0;
    unsigned long long nf = 0;
    for (int y = blockIdx.x; y < Ny; y += gridDim.x) {
        const int yp = y + 1 == Ny ? 0 : y + 1, ym = y == 0 ? Ny - 1 : y - 1;
        const size_t r = size_t(y) * Nx;
        // A thread's sites of one row (at most ceil(Nx / DIAG_THREADS) terms of
        // equal sign) are summed plainly in FP64; the row sums enter the
        // compensated sums. The FP64 pipe is the bound of this kernel, so
        // per-site work is kept to the squares and one add per sum.
        double erow = 0.0, drow = 0.0;
        for (int x = threadIdx.x; x < Nx; x += blockDim.x) {
            const size_t i = r + x;
            double sq[6];
#pragma unroll
            for (int c = 0; c < 6; ++c) {
                const T v = q[size_t(c) * P + i];
                if (!finite_val(v)) ++nf;
                const double dv = double(v);
                sq[c] = dv * dv;
            }
            const double b2 = sq[3] + sq[4] + sq[5];
            erow += (sq[0] + sq[1] + sq[2]) + b2;
            b2max = fmax(b2max, b2);
            const int xp = x + 1 == Nx ? 0 : x + 1, xm = x == 0 ? Nx - 1 : x - 1;
            const double dv = 0.5 * (double(q3[r + xp]) - double(q3[r + xm])) +
                              0.5 * (double(q4[size_t(yp) * Nx + x]) - double(q4[size_t(ym) * Nx + x]));
            drow = fma(dv, dv, drow);
            dmax = fmax(dmax, fabs(dv));
        }
        e.add(erow);
        d.add(drow);
    }
    const double bmax = sqrt(b2max);  // sqrt is monotonic: the max of the site norms
    block_reduce_write(Partial{e.s, e.c, d.s, d.c, dmax, bmax, nf, 0ull}, part);
}

// Exact FP32 -> FP64 conversion on the integer pipe (this kernel is bound by
// GB300's FP64 pipe, which also executes the hardware conversion): zero and
// normal values by rebiasing the exponent and widening the mantissa; subnormal,
// infinite and NaN values take the hardware conversion.
__device__ __forceinline__ double f2d_exact(float v) {
    const unsigned u = __float_as_uint(v);
    const unsigned e = (u >> 23) & 0xffu;
    const bool zero = (u << 1) == 0u;
    if (zero || e - 1u < 254u) {
        const unsigned mag = zero ? 0u : (((e + 896u) << 20) | ((u >> 3) & 0xfffffu));
        return __hiloint2double(int((u & 0x80000000u) | mag), zero ? 0 : int(u << 29));
    }
    return double(v);
}

// Unevaluated FP32 pair hi + lo (|lo| about 2^-24 |hi|). The rounding intrinsics
// keep the compiler from contracting the error terms away.
struct FPair {
    float hi, lo;
    // adds the pair (p, e): the high parts by TwoSum, the low parts in FP32
    __device__ __forceinline__ void add(float p, float e) {
        const float s = __fadd_rn(hi, p);
        const float bb = __fsub_rn(s, hi);
        const float t = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(p, bb));
        lo = __fadd_rn(lo, __fadd_rn(t, e));
        hi = s;
    }
    __device__ __forceinline__ double value() const { return f2d_exact(hi) + f2d_exact(lo); }
};

// Screening of a maximum by FP32 approximations f >= 0 of the FP64 values
// (relative error below 2^-20): a site above the pending one by more than
// 2^-18 replaces it, a site below it by more is dropped, and only one in
// between has its FP64 value computed at once; the pending site's is at the
// end. (Computing it whenever a running maximum rose did so at a third of the
// sites of a smooth field, for some lane of the warp.)
struct Screen {
    float best = 0.0f;
    __device__ __forceinline__ bool replaces(float f) const { return f > best * (1.0f + 0x1p-18f); }
    __device__ __forceinline__ bool close(float f) const { return f >= best * (1.0f - 0x1p-18f) && f > 0.0f; }
};

// |v| in [2^-50, 2^60): a square and its FMA error are then normal FP32 numbers
// or the error is zero, and sums of squares do not overflow.
__device__ __forceinline__ bool pair_range(float v) {
    return (__float_as_uint(v) & 0x7fffffffu) - 0x26800000u < 0x37000000u;
}
__device__ __forceinline__ bool is_zero(float v) { return (__float_as_uint(v) << 1) == 0u; }

// Sum of squares of six values below 2^60, the largest zero or at least 2^-44
// (a square of less than 2^-100 has an error term off by 2^-149 at most).
__device__ __forceinline__ FPair sum_of_squares(const float (&v)[6]) {
    FPair s;
    s.hi = __fmul_rn(v[0], v[0]);
    s.lo = __fmaf_rn(v[0], v[0], -s.hi);
#pragma unroll
    for (int c = 1; c < 6; ++c) {
        const float p = __fmul_rn(v[c], v[c]);
        s.add(p, __fmaf_rn(v[c], v[c], -p));
    }
    return s;
}

// div B of a site, times 2: (r - l) + (u - d) as the FP64 operations give it (each
// is exact, or rounds once). The differences, their sum and all of their errors are
// formed in FP32 (TwoSum); where the errors add up exactly (values within about 2^23
// of each other) the sum of the two parts is the only FP64 operation, and there is
// none where the FP32 sum is exact.
__device__ __forceinline__ double divergence(float r, float l, float u, float d) {
    const float h1 = __fsub_rn(r, l), b1 = __fsub_rn(h1, r);
    const float e1 = __fsub_rn(__fsub_rn(r, __fsub_rn(h1, b1)), __fadd_rn(l, b1));
    const float h2 = __fsub_rn(u, d), b2 = __fsub_rn(h2, u);
    const float e2 = __fsub_rn(__fsub_rn(u, __fsub_rn(h2, b2)), __fadd_rn(d, b2));
    const float s = __fadd_rn(h1, h2), bs = __fsub_rn(s, h1);
    const float t = __fadd_rn(__fsub_rn(h1, __fsub_rn(s, bs)), __fsub_rn(h2, bs));
    const float te = __fadd_rn(t, e2), lo = __fadd_rn(te, e1);
    // both sums exact (so their TwoSum errors vanish), and no overflow, infinity or NaN
    if (fabsf(s) < 0x1p120f && __fsub_rn(te, t) == e2 && __fsub_rn(te, e2) == t && __fsub_rn(lo, te) == e1 &&
        __fsub_rn(lo, e1) == te) {
        const double v = f2d_exact(s);
        return lo == 0.0f ? v : v + f2d_exact(lo);
    }
    return (f2d_exact(r) - f2d_exact(l)) + (f2d_exact(u) - f2d_exact(d));
}

// FP32 state. GB300's FP64 pipe takes a warp instruction in 64 cycles of a
// scheduler (the generic kernel below is bound by it, and so was this one with
// six FP64 operations per site: 305 us at 4096^2), so a site costs few:
//  * its sum of squares is an FP32 pair (products with their FMA errors, sums by
//    TwoSum), added to a pair that enters the FP64 sum after PAIR_SITES sites:
//    relative error about 2^-46 of such a partial sum, over many of them below that
//    of the squares' own low parts (2^-50, all of one sign: the low bits of a square
//    are not uniform);
//  * the divergence (see above) enters the FP64 sum by one FMA, two operations at
//    most (as a pair squared in FP32 the sum was off by 5 to 8 units of 2^-53, in
//    FP64 by less than one); the factors 1/2 and 1/4 are applied to the reduced max
//    and sum;
//  * max |B| is screened in FP32 (Screen below); max |div| is kept as the bit
//    pattern of a non-negative double (integer order = numeric order; NaN
//    excluded, as fmax would).
// Sites with a value outside [2^-60, 2^60) take FP64 for their squares, those with no
// value of 2^-44 or more (squares near FP32's smallest) a pair of scaled values that
// enters the FP64 sum at once.
constexpr int PAIR_SITES = 32;
// (four blocks per SM: all of the grid's 608 resident at once)
__global__ void __launch_bounds__(DIAG_THREADS, 4) diag_partial_f32(const float *__restrict__ q, int Nx, int Ny,
                                                                 Partial *__restrict__ part) {
    const size_t P = size_t(Nx) * size_t(Ny);
    const float *q4 = q + 4 * P;
    CSum e{0.0, 0.0}, d{0.0, 0.0};
    unsigned long long dmax_bits = 0;
    double b2max = 0.0;
    Screen sb, st;  // st: sites with |B|^2 < 2^-116, values scaled by 2^90
    bool tiny_pending = false;
    float pb[3] = {0.0f, 0.0f, 0.0f};  // the pending site's values
    auto exact_b2 = [&](float v3, float v4, float v5) {
        const double d3 = f2d_exact(v3), d4 = f2d_exact(v4), d5 = f2d_exact(v5);
        const double b2 = (d3 * d3 + d4 * d4) + d5 * d5;
        if (b2 > b2max) b2max = b2;
    };
    unsigned long long nf = 0;
    FPair ep{0.0f, 0.0f};
    double e64 = 0.0, d64 = 0.0;  // plain sums of the pending sites
    int pending = 0;
    const unsigned W = unsigned(Nx);
    for (int y = blockIdx.x; y < Ny; y += gridDim.x) {
        const int yp = y + 1 == Ny ? 0 : y + 1, ym = y == 0 ? Ny - 1 : y - 1;
        const float *row[6];
#pragma unroll
        for (int c = 0; c < 6; ++c) row[c] = q + c * P + size_t(y) * W;
        const float *const q4p = q4 + size_t(yp) * W, *const q4m = q4 + size_t(ym) * W;
        for (unsigned x = threadIdx.x; x < W; x += DIAG_THREADS) {
            const unsigned xp = x + 1 == W ? 0 : x + 1, xm = x == 0 ? W - 1 : x - 1;
            float v[6];
            unsigned big[2] = {0u, 0u}, small = 0xffffffffu;  // big: of Q0-Q2, of B
#pragma unroll
            for (int c = 0; c < 6; ++c) {
                v[c] = row[c][x];
                const unsigned ua = __float_as_uint(v[c]) & 0x7fffffffu;
                big[c / 3] = max(big[c / 3], ua);
                small = min(small, ua - 1u);  // zero counts as large
            }
            const unsigned bigq = max(big[0], big[1]);
            const float l = row[3][xm], rr = row[3][xp], dn = q4m[x], up = q4p[x];
            if (bigq < 0x5d800000u && small >= 0x217fffffu) {  // every |v| zero or in [2^-60, 2^60)
                if (bigq - 1u >= 0x297fffffu) {  // the largest zero or at least 2^-44
                    const FPair s = sum_of_squares(v);
                    ep.add(s.hi, s.lo);
                } else {
                    float w[6];
#pragma unroll
                    for (int c = 0; c < 6; ++c) w[c] = v[c] * 0x1p64f;
                    const FPair s = sum_of_squares(w);
                    e64 = fma(f2d_exact(s.hi), 0x1p-128, e64);
                    e64 = fma(f2d_exact(s.lo), 0x1p-128, e64);
                }
            } else {
#pragma unroll
                for (int c = 0; c < 6; ++c) {
                    if (!isfinite(v[c])) ++nf;
                    const double dv = f2d_exact(v[c]);
                    e64 = fma(dv, dv, e64);
                }
            }
            // max |B|: the pending site is one of tiny values only while no other was met
            const float b2f = fmaf(v[3], v[3], fmaf(v[4], v[4], v[5] * v[5]));
            if (big[1] >= 0x5d800000u) {
                exact_b2(v[3], v[4], v[5]);
            } else if (b2f >= 0x1p-116f) {
                if (sb.replaces(b2f)) {
                    if (tiny_pending && b2f < 0x1p-115f) exact_b2(pb[0], pb[1], pb[2]);
                    tiny_pending = false;
                    sb.best = b2f;
                    pb[0] = v[3]; pb[1] = v[4]; pb[2] = v[5];
                } else if (sb.close(b2f) && !(v[3] == pb[0] && v[4] == pb[1] && v[5] == pb[2])) {
                    exact_b2(v[3], v[4], v[5]);
                }
            } else if (big[1] != 0u && sb.best < 0x1p-115f) {
                const float w3 = v[3] * 0x1p90f, w4 = v[4] * 0x1p90f, w5 = v[5] * 0x1p90f;
                const float t2f = fmaf(w3, w3, fmaf(w4, w4, w5 * w5));
                if (sb.best > 0.0f) {
                    exact_b2(v[3], v[4], v[5]);
                } else if (st.replaces(t2f)) {
                    tiny_pending = true;
                    st.best = t2f;
                    pb[0] = v[3]; pb[1] = v[4]; pb[2] = v[5];
                } else if (st.close(t2f) && !(v[3] == pb[0] && v[4] == pb[1] && v[5] == pb[2])) {
                    exact_b2(v[3], v[4], v[5]);
                }
            }
            // the divergence: in FP32 where its parts add up exactly, otherwise in FP64
            const double dv = divergence(rr, l, up, dn);
            d64 = fma(dv, dv, d64);
            const unsigned long long ab = static_cast<unsigned long long>(__double_as_longlong(dv)) & 0x7fffffffffffffffull;
            if (ab <= 0x7ff0000000000000ull && ab > dmax_bits) dmax_bits = ab;
            if (++pending == PAIR_SITES) {
                e.add(ep.value() + e64);
                d.add(0.25 * d64);
                ep = FPair{0.0f, 0.0f};
                e64 = d64 = 0.0;
                pending = 0;
            }
        }
    }
    e.add(ep.value() + e64);
    d.add(0.25 * d64);
    exact_b2(pb[0], pb[1], pb[2]);
    const double dmax = 0.5 * __longlong_as_double(static_cast<long long>(dmax_bits));
    block_reduce_write(Partial{e.s, e.c, d.s, d.c, dmax, sqrt(b2max), nf, 0ull}, part);
}

// Divergence of D (Sec. 4.2): D = (n_x q0, n_y q1, n_z q2) for the diagonal
// dielectric eps_i = n_i^2 (Eq. 15: q_i = n_i E_i), central differences in
// lattice units. The record's div fields hold sum div^2 and max |div|, its B
// field max |D|; the energy fields are zero.
//
// The FP64 pipe is the bound, so each product is formed once: a warp covers 30
// columns with one more on either side (D_x of the neighbours by shuffle) and
// walks down a tile's rows (D_y of the rows above and below in registers): six
// FP64 operations per site and those of the tiles' halo rows, shared columns and
// maxima, 8.6 by the pipe's time (4096^2: 298 us, pipe 82% busy), where a thread per
// site that formed its four neighbours' products and |D|^2 itself took about thirty
// (760 us).
// max |D|^2 is screened in FP32 (Screen), FP32 states are widened
// on the integer pipe, and the factors 1/2 and 1/4 are applied to the reduced
// values.
constexpr int DIVD_COLS = 30 * (DIAG_THREADS / 32);
constexpr int DIVD_MAX_ROWS = 32;

__device__ __forceinline__ bool same_bits(double a, double b) {
    return __double_as_longlong(a) == __double_as_longlong(b);
}
__device__ __forceinline__ double widen(float v) { return f2d_exact(v); }
__device__ __forceinline__ double widen(double v) { return v; }
// v truncated to FP32 on the integer pipe; *ok is cleared unless v is zero or
// |v| in [2^-50, 2^60) (then the result is within 2^-22 of v, relatively).
__device__ __forceinline__ float narrow_for_screen(double v, bool *ok) {
    const unsigned hi = unsigned(__double2hiint(v)), lo = unsigned(__double2loint(v));
    const unsigned ex = (hi >> 20) & 0x7ffu;
    const bool zero = ((hi << 1) | lo) == 0u;
    *ok = *ok && (zero || ex - (1023u - 50u) < 110u);
    return zero ? 0.0f : __uint_as_float((hi & 0x80000000u) | ((ex - 896u) << 23) | ((hi & 0xfffffu) << 3) | (lo >> 29));
}

template <typename T>
__global__ void __launch_bounds__(DIAG_THREADS, 4) divD_partial(const T *__restrict__ q, const double *__restrict__ idx,
                                                             int Nx, int Ny, int tile_rows,
                                                             Partial *__restrict__ part) {
    const size_t P = size_t(Nx) * size_t(Ny);
    const T *q0 = q, *q1 = q + P, *q2 = q + 2 * P;
    const double *nx = idx, *ny = idx + P, *nz = idx + 2 * P;
    CSum d{0.0, 0.0};
    unsigned long long dmax_bits = 0;
    double d2max = 0.0;
    Screen sc;
    double pdx = 0.0, pdy = 0.0, pnz = 0.0;  // the pending site's D_x, D_y, n_z
    T pv2 = T(0);
    auto exact_d2 = [&](double dx, double dy, double n, T v) {
        const double dz = n * widen(v);
        const double d2 = dx * dx + dy * dy + dz * dz;
        if (d2 > d2max) d2max = d2;
    };
    unsigned long long nf = 0;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int ctiles = (Nx + DIVD_COLS - 1) / DIVD_COLS, rtiles = (Ny + tile_rows - 1) / tile_rows;
    for (long long t = blockIdx.x; t < (long long)ctiles * rtiles; t += gridDim.x) {
        const int xc = int(t % ctiles) * DIVD_COLS + warp * 30 + lane - 1;
        const int y0 = int(t / ctiles) * tile_rows, y1 = min(y0 + tile_rows, Ny);
        const bool mine = lane >= 1 && lane <= 30 && xc < Nx;
        int x = xc % Nx;  // halo columns wrap around; columns past them are not used
        x = x < 0 ? x + Nx : x;
        auto dy_of = [&](int y) {
            const int w = y < 0 ? y + Ny : (y >= Ny ? y - Ny : y);
            const size_t i = size_t(w) * Nx + x;
            return ny[i] * widen(q1[i]);
        };
        double below = dy_of(y0 - 1), here = dy_of(y0), sum = 0.0;
        for (int y = y0; y < y1; ++y) {
            const size_t i = size_t(y) * Nx + x;
            const T v0 = q0[i], v1 = q1[i], v2 = q2[i];
            const double above = dy_of(y + 1);
            const double dx = nx[i] * widen(v0);
            const double left = __shfl_up_sync(0xffffffffu, dx, 1), right = __shfl_down_sync(0xffffffffu, dx, 1);
            const double dv = (right - left) + (above - below);
            sum = fma(dv, dv, sum);  // (lanes whose column is another warp's do not add theirs)
            const unsigned long long ab = static_cast<unsigned long long>(__double_as_longlong(dv)) &
                                          0x7fffffffffffffffull;
            if (mine) {
                if (ab <= 0x7ff0000000000000ull && ab > dmax_bits) dmax_bits = ab;
                if (!finite_val(v0) || !finite_val(v1) || !finite_val(v2)) ++nf;
            }
            bool ok = true;
            const double dnz = nz[i];
            const float fx = narrow_for_screen(dx, &ok), fy = narrow_for_screen(here, &ok);
            const float fz = narrow_for_screen(dnz, &ok) * narrow_for_screen(widen(v2), &ok);
            ok = ok && (is_zero(fz) || pair_range(fz));  // D_z itself, as D_x and D_y are products above
            const float f = fmaf(fx, fx, fmaf(fy, fy, fz * fz));
            if (mine) {
                if (!ok) {
                    exact_d2(dx, here, dnz, v2);
                } else if (sc.replaces(f)) {
                    sc.best = f;
                    pdx = dx;
                    pdy = here;
                    pnz = dnz;
                    pv2 = v2;
                } else if (sc.close(f) && !(same_bits(dx, pdx) && same_bits(here, pdy) && same_bits(dnz, pnz) &&
                                            v2 == pv2)) {
                    exact_d2(dx, here, dnz, v2);
                }
            }
            below = here;
            here = above;
        }
        if (mine) d.add(0.25 * sum);
    }
    exact_d2(pdx, pdy, pnz, pv2);
    const double dmax = 0.5 * __longlong_as_double(static_cast<long long>(dmax_bits));
    block_reduce_write(Partial{0.0, 0.0, d.s, d.c, dmax, sqrt(d2max), nf, 0ull}, part);
}

// One block combines the partial records in a fixed tree: half of its warps the
// energy sums (and max |div|, the non-finite count), the other half the
// divergence sums (and max |B|), lanes by shuffle. Latency is all it costs, a
// chain of FP64 additions per level (both sums in every thread, through shared
// memory: 13 us).
__global__ void __launch_bounds__(DIAG_THREADS) diag_final(const Partial *__restrict__ part, int n,
                                                           DiagResult *__restrict__ out) {
    constexpr int HALF = DIAG_THREADS / 2, WARPS = HALF / 32;
    const bool first = threadIdx.x < HALF;
    CSum s{0.0, 0.0};
    double mx = 0.0;
    unsigned long long nf = 0;
    for (int i = int(threadIdx.x % HALF); i < n; i += HALF) {
        const Partial p = part[i];
        s.merge(first ? CSum{p.e_s, p.e_c} : CSum{p.d_s, p.d_c});
        const double m = first ? p.dmax : p.bmax;  // non-negative or NaN: the larger number
        mx = m > mx ? m : mx;
        nf += p.nonfinite;
    }
    for (int o = 16; o > 0; o >>= 1) {
        s.merge(CSum{__shfl_down_sync(0xffffffffu, s.s, o), __shfl_down_sync(0xffffffffu, s.c, o)});
        const double m = __shfl_down_sync(0xffffffffu, mx, o);
        mx = m > mx ? m : mx;
        nf += __shfl_down_sync(0xffffffffu, nf, o);
    }
    __shared__ CSum ss[2 * WARPS];
    __shared__ double sm[2 * WARPS];
    __shared__ unsigned long long sn[2 * WARPS];
    const int w = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) {
        ss[w] = s;
        sm[w] = mx;
        sn[w] = nf;
    }
    __syncthreads();
    if (threadIdx.x % HALF == 0) {
        for (int k = 1; k < WARPS; ++k) {
            s.merge(ss[w + k]);
            mx = sm[w + k] > mx ? sm[w + k] : mx;
            nf += sn[w + k];
        }
        if (first) {
            out->energy_sum = s.s + s.c;
            out->div_max = mx;
            out->nonfinite = nf;
        } else {
            out->div_sq_sum = s.s + s.c;
            out->b_max = mx;
        }
    }
}

}  // namespace

int diag_blocks(int Nx, int Ny) {
    (void)Nx;
    return Ny < 4 * 152 ? Ny : 4 * 152;
}

size_t diag_scratch_bytes(int Nx, int Ny) {
    return size_t(diag_blocks(Nx, Ny)) * sizeof(Partial) + 256;
}

cudaError_t launch_diagnostics(const void *q, int precision, int Nx, int Ny, void *scratch, DiagResult *out_dev,
                               cudaStream_t st) {
    const int G = diag_blocks(Nx, Ny);
    Partial *part = static_cast<Partial *>(scratch);
    if (precision == 0)
        diag_partial_f32<<<G, DIAG_THREADS, 0, st>>>(static_cast<const float *>(q), Nx, Ny, part);
    else
        diag_partial<double><<<G, DIAG_THREADS, 0, st>>>(static_cast<const double *>(q), Nx, Ny, part);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    diag_final<<<1, DIAG_THREADS, 0, st>>>(part, G, out_dev);
    return cudaGetLastError();
}

cudaError_t launch_divD(const void *q, int precision, const double *index, int Nx, int Ny, void *scratch,
                        DiagResult *out_dev, cudaStream_t st) {
    // tiles of at most 32 rows, lower where that would leave blocks idle
    const int ctiles = (Nx + DIVD_COLS - 1) / DIVD_COLS;
    int rows = int((long long)ctiles * Ny / diag_blocks(Nx, Ny));
    rows = rows < 4 ? 4 : (rows > DIVD_MAX_ROWS ? DIVD_MAX_ROWS : rows);
    const long long tiles = (long long)ctiles * ((Ny + rows - 1) / rows);
    const int G = tiles < diag_blocks(Nx, Ny) ? int(tiles) : diag_blocks(Nx, Ny);
    Partial *part = static_cast<Partial *>(scratch);
    if (precision == 0)
        divD_partial<float><<<G, DIAG_THREADS, 0, st>>>(static_cast<const float *>(q), index, Nx, Ny, rows, part);
    else
        divD_partial<double><<<G, DIAG_THREADS, 0, st>>>(static_cast<const double *>(q), index, Nx, Ny, rows, part);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    diag_final<<<1, DIAG_THREADS, 0, st>>>(part, G, out_dev);
    return cudaGetLastError();
}

}  // namespace qla

// ---------------------------------------------------------------------------
// Allocation-free diagnostics (qla_diagnostics_noalloc in include/qla.h).
//
// Some callers cannot allocate device memory at the point where they need
// the diagnostics: an application that hands all of the GPU's memory to its
// own allocator up front (a framework's caching pool, a fixed budget per job)
// and forbids cudaMalloc afterwards, or a monitoring loop that must not block
// on the allocator or fail with out-of-memory halfway through a long run. This variant
// runs the same two reduction kernels as the context-based diagnostics, but
// keeps their scratch (the per-block partial records and the final result) in
// the file-scope device array below instead of memory from cudaMalloc.
//
// The array is reserved in every GPU that loads the library, for the life of
// the process. All calls share it and it keeps the previous call's contents:
// every record a call reads is written earlier in the same call, so nothing
// has to be cleared, but two calls whose kernels overlap on the GPU (different
// streams, or different host threads) race on it.
// ---------------------------------------------------------------------------
#include <limits.h>

#include "../../include/qla.h"

namespace qla {
namespace {

constexpr int NOALLOC_ROWS_PER_BLOCK = 4;
constexpr int NOALLOC_MAX_PARTIALS = 4096;  // lattices of at most 4096 * 4 = 16384 rows
struct NoallocScratch {
    Partial part[NOALLOC_MAX_PARTIALS];
    DiagResult result;
};

static __device__ __align__(256) NoallocScratch g_noalloc_scratch;

// Device address of the array on the current device. In host code the
// symbol g_noalloc_scratch is only a host-side stand-in, so the address is
// looked up on every call: a cached address would go stale after a device
// reset or a re-created primary context, when the module reloads elsewhere.
// The first call on a device may load the module: make it before any stream
// capture.
cudaError_t noalloc_scratch(NoallocScratch **out) {
    void *p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess) return e;
    *out = static_cast<NoallocScratch *>(p);
    return cudaSuccess;
}

}  // namespace
}  // namespace qla

extern "C" qla_status qla_diagnostics_noalloc(const void *q, int precision, int Nx, int Ny, void *stream,
                                              qla_diag *out) {
    using namespace qla;
    if (!q || !out || Nx < 1 || Ny < 1 || (long long)Nx * (long long)Ny > INT_MAX ||
        (precision != QLA_FP32 && precision != QLA_FP64))
        return QLA_EINVAL;
    const int G = (Ny + NOALLOC_ROWS_PER_BLOCK - 1) / NOALLOC_ROWS_PER_BLOCK;
    if (G > NOALLOC_MAX_PARTIALS) return QLA_EINVAL;  // Ny above 16384: the static scratch is too small
    NoallocScratch *s = nullptr;
    if (noalloc_scratch(&s) != cudaSuccess) {
        cudaGetLastError();
        return QLA_ECUDA;
    }
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (precision == QLA_FP32)
        diag_partial_f32<<<G, DIAG_THREADS, 0, st>>>(static_cast<const float *>(q), Nx, Ny, s->part);
    else
        diag_partial<double><<<G, DIAG_THREADS, 0, st>>>(static_cast<const double *>(q), Nx, Ny, s->part);
    if (cudaGetLastError() != cudaSuccess) return QLA_ECUDA;
    diag_final<<<1, DIAG_THREADS, 0, st>>>(s->part, G, &s->result);
    if (cudaGetLastError() != cudaSuccess) return QLA_ECUDA;
    DiagResult r;
    if (cudaMemcpyAsync(&r, &s->result, sizeof(r), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess) {
        cudaGetLastError();
        return QLA_ECUDA;
    }
    out->energy = r.energy_sum / (double(Nx) * double(Ny));
    out->div_l2_sq = r.div_sq_sum;
    out->div_max = r.div_max;
    out->b_max = r.b_max;
    out->nonfinite = (long long)r.nonfinite;
    return r.nonfinite ? QLA_ENONFINITE : QLA_OK;
}
