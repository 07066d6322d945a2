// Set-up kernels: rotation/potential coefficients (Eq. 24-25), the pulse
// initial condition and precision conversions.
#include <math.h>

#include <algorithm>
#include <cmath>

#include "qla_internal.h"

namespace qla {

namespace {

// FP32 rotation pair (t, s): t = tan(a / 2) rounded to FP32, and s the FP32 value
// nearest to 2t / (1 + t^2), the sine of the angle 2 atan(t) that t represents
// exactly. The three shears and the four-operation form of the sweep (determinant
// exactly 1) are then a rotation to within one rounding of s, and the angle
// differs from a by at most half an ulp of t.
__device__ void rotation_pair_f32(double ang, float &tf, float &sf) {
    tf = (float)tan(0.5 * ang);
    const double t = (double)tf;
    sf = (float)(2.0 * t / (1.0 + t * t));
}

// FP32 (cos(a) - 1, sin(a)) pair chosen among FP32 values within a few ulps of
// the correctly rounded ones so that (1 + m)^2 + s^2 - 1 (evaluated exactly in
// FP64: every term is a product of two FP32 values) is as small as possible:
// each rotation then keeps the energy (Eq. 27) closely, with the angle changed
// by a few ulps of m and s at most.
__device__ void wide_pair_f32(double ang, float &mf, float &sf) {
    const double sh = sin(0.5 * ang);
    mf = (float)(-2.0 * sh * sh);  // cos(ang) - 1 without cancellation
    sf = (float)sin(ang);
    if (!(fabsf(mf) >= 1e-30f) || !(fabsf(sf) >= 1e-30f)) return;  // zero or nearly: the rounded values
    const int mi = __float_as_int(mf), si = __float_as_int(sf);
    double best = 1e300;
    int bdm = 0, bds = 0;
    for (int dm = -4; dm <= 4; ++dm) {
        for (int ds = -2; ds <= 2; ++ds) {
            const double m = (double)__int_as_float(mi + dm), s = (double)__int_as_float(si + ds);
            const double e = fabs(2.0 * m + m * m + s * s);
            if (e < best || (e == best && abs(dm) + abs(ds) < abs(bdm) + abs(bds))) {
                best = e;
                bdm = dm;
                bds = ds;
            }
        }
    }
    mf = __int_as_float(mi + bdm);
    sf = __int_as_float(si + bds);
}

// How a pair is stored (see CoefPair and rot in the sweep): a rotation
// (tan(a/2), sin a), one in the form for any angle (cos a - 1, sin a), or a
// printed potential row (cos a - 1, sin a).
enum PairKind { PK_ROTATION, PK_WIDE, PK_PRINTED_V };
__device__ __forceinline__ PairKind rotation_kind(int mode) { return mode & MODE_WIDE ? PK_WIDE : PK_ROTATION; }

template <typename T>
__device__ void make_pair_of(double ang, PairKind kind, T &x, T &y) {
    if (sizeof(T) == 4 && kind == PK_WIDE) {
        float m, sn;
        wide_pair_f32(ang, m, sn);
        x = m;
        y = sn;
    } else if (kind != PK_ROTATION) {
        const double sh = sin(0.5 * ang);
        x = (T)(-2.0 * sh * sh);  // cos(ang) - 1 without cancellation
        y = (T)sin(ang);
    } else if constexpr (sizeof(T) == 4) {
        rotation_pair_f32(ang, x, y);
    } else {
        x = tan(0.5 * ang);
        y = sin(ang);
    }
}

template <typename T>
__device__ void store_pair(T *coef, size_t P, int pair, size_t i, double ang, PairKind kind) {
    T *dst = coef + 2 * (size_t(pair) * P + i);
    make_pair_of<T>(ang, kind, dst[0], dst[1]);
}

// Eq. 25 at site (x, y), central differences over lattice spacing delta:
// delta^2 (dn/dx) / n^2 along x (axis 0) or y (axis 1).
__device__ __forceinline__ double potential_angle(const double *__restrict__ n, int x, int y, int Nx, int Ny, int axis,
                                                  double delta) {
    const int xp = x + 1 == Nx ? 0 : x + 1, xm = x == 0 ? Nx - 1 : x - 1;
    const int yp = y + 1 == Ny ? 0 : y + 1, ym = y == 0 ? Ny - 1 : y - 1;
    const size_t r = size_t(y) * Nx;
    const double v = n[r + x];
    const double d = axis == 0 ? (n[r + xp] - n[r + xm]) / (2.0 * delta)
                               : (n[size_t(yp) * Nx + x] - n[size_t(ym) * Nx + x]) / (2.0 * delta);
    return delta * delta * d / (v * v);
}

// One thread per site. n: [3][Ny][Nx] double (n_x, n_y, n_z).
template <typename T>
__global__ void coef_kernel(const double *__restrict__ n, T *__restrict__ coef, int Nx, int Ny, double delta,
                            int interleaved, int mode) {
    const size_t P = size_t(Nx) * size_t(Ny);
    const double *nx = n, *ny = n + P, *nz = n + 2 * P;
    // effective potential angle: halved when interleaved (Eq. 28), halved
    // again for the unitary pair rotation
    const double vscale = (interleaved ? 0.5 : 1.0) * (mode & MODE_UNITARY ? 0.5 : 1.0);
    for (size_t i = blockIdx.x * size_t(blockDim.x) + threadIdx.x; i < P; i += size_t(gridDim.x) * blockDim.x) {
        const int y = int(i / Nx), x = int(i % Nx);
        // Eq. 24
        const double th0 = delta / (4.0 * nx[i]), th1 = delta / (4.0 * ny[i]), th2 = delta / (4.0 * nz[i]);
        const double b0 = potential_angle(ny, x, y, Nx, Ny, 0, delta);
        const double b1 = potential_angle(nx, x, y, Nx, Ny, 1, delta);
        const double b2 = potential_angle(nz, x, y, Nx, Ny, 0, delta);
        const double b3 = potential_angle(nz, x, y, Nx, Ny, 1, delta);
        const PairKind ck = rotation_kind(mode), vk = mode & MODE_UNITARY ? ck : PK_PRINTED_V;
        store_pair<T>(coef, P, P_TM_C, i, th2, ck);
        store_pair<T>(coef, P, P_TE_CX, i, th1, ck);
        store_pair<T>(coef, P, P_TE_CY, i, th0, ck);
        store_pair<T>(coef, P, P_TM_VX, i, b2 * vscale, vk);
        store_pair<T>(coef, P, P_TM_VY, i, b3 * vscale, vk);
        store_pair<T>(coef, P, P_TE_VX, i, b0 * vscale, vk);
        store_pair<T>(coef, P, P_TE_VY, i, b1 * vscale, vk);
    }
}

// The same pairs as the marching form's records (one block per row of a strip).
template <typename T>
__global__ void march_records_kernel(const double *__restrict__ n, T *__restrict__ rec, int fam, MarchGeo g,
                                     double delta, int interleaved, int mode) {
    const size_t P = size_t(g.Nx) * size_t(g.Ny);
    const double *nx = n, *ny = n + P, *nz = n + 2 * P;
    const double *ncx = fam ? ny : nz, *ncy = fam ? nx : nz;  // indices of C_X and V_X, of C_Y and V_Y
    const double vscale = (interleaved ? 0.5 : 1.0) * (mode & MODE_UNITARY ? 0.5 : 1.0);
    const PairKind ck = rotation_kind(mode), vk = mode & MODE_UNITARY ? ck : PK_PRINTED_V;
    const int rows = MARCH_ABOVE + g.Ny + MARCH_BELOW, strip = blockIdx.x;
    for (int r = blockIdx.y; r < rows; r += gridDim.y) {
        int y = (r - MARCH_ABOVE) % g.Ny;
        y = y < 0 ? y + g.Ny : y;
        for (int c = threadIdx.x; c < g.W; c += blockDim.x) {
            int x = (strip * g.w_valid - g.halo + c) % g.Nx;
            x = x < 0 ? x + g.Nx : x;
            const size_t i = size_t(y) * g.Nx + x;
            T *const d = rec + (size_t(strip) * rows + r) * MARCH_FIELDS * g.W +
                         march_column(c, int(sizeof(T)));
            make_pair_of<T>(delta / (4.0 * ncx[i]), ck, d[F_CX * g.W], d[(F_CX + 1) * g.W]);
            if (fam) make_pair_of<T>(delta / (4.0 * ncy[i]), ck, d[F_CY * g.W], d[(F_CY + 1) * g.W]);
            for (int axis = 0; axis < 2; ++axis) {
                const double b = potential_angle(axis ? ncy : ncx, x, y, g.Nx, g.Ny, axis, delta) * vscale;
                T *const v = d + (axis ? F_VY : F_VX) * g.W;
                if (b == 0.0) {  // the pair of a zero angle, without its sines
                    v[0] = T(-0.0);
                    v[g.W] = T(b);
                } else {
                    make_pair_of<T>(b, vk, v[0], v[g.W]);
                }
            }
        }
    }
}

// flags[strip][r] (MARCH_V, MARCH_C): whether any V pair of the strip's columns
// is nonzero in rows [r - march_flag_back(2), r + MARCH_GROUP - 1], and whether
// any C pair of rows [r - MARCH_SAME_BACK, r + MARCH_SAME_AHEAD] differs from the
// row above it.
constexpr int FLAG_ROWS = 64;
template <typename T>
__global__ void __launch_bounds__(256) march_flags_kernel(const T *__restrict__ rec, unsigned char *__restrict__ flags,
                                                          int fam, MarchGeo g) {
    constexpr int BACK = march_flag_back(2) > MARCH_SAME_BACK ? march_flag_back(2) : MARCH_SAME_BACK;
    constexpr int AHEAD = MARCH_GROUP - 1 > MARCH_SAME_AHEAD ? MARCH_GROUP - 1 : MARCH_SAME_AHEAD;
    __shared__ unsigned char rf[FLAG_ROWS + BACK + AHEAD];
    const int strip = blockIdx.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int rows = MARCH_ABOVE + g.Ny + MARCH_BELOW;
    const int cfields = fam ? 4 : 2;  // TM: C_Y is not stored
    static_assert(BACK < MARCH_ABOVE && AHEAD < MARCH_BELOW && F_CX == 0 && F_CY == 2, "rows and fields compared");
    for (int r0 = blockIdx.y * FLAG_ROWS; r0 < g.Ny; r0 += gridDim.y * FLAG_ROWS) {
        const int n = min(FLAG_ROWS, g.Ny - r0);
        for (int k = warp; k < n + BACK + AHEAD; k += 8) {
            const T *const r = rec + (size_t(strip) * rows + MARCH_ABOVE + r0 - BACK + k) * MARCH_FIELDS * g.W;
            const T *const above = r - MARCH_FIELDS * g.W;
            bool nz = false, differs = false;
            for (int c = lane; c < 4 * g.W; c += 32) nz = nz || r[F_VX * g.W + c] != T(0);
            for (int c = lane; c < cfields * g.W; c += 32) differs = differs || r[c] != above[c];
            nz = __any_sync(0xffffffffu, nz);
            differs = __any_sync(0xffffffffu, differs);
            if (lane == 0) rf[k] = (unsigned char)((nz ? MARCH_V : 0) | (differs ? MARCH_C : 0));
        }
        __syncthreads();
        for (int k = threadIdx.x; k < n; k += 256) {
            unsigned f = 0;
            for (int i = -march_flag_back(2); i < MARCH_GROUP; ++i) f |= rf[k + BACK + i] & MARCH_V;
            for (int i = -MARCH_SAME_BACK; i <= MARCH_SAME_AHEAD; ++i) f |= rf[k + BACK + i] & MARCH_C;
            flags[size_t(strip) * g.Ny + r0 + k] = (unsigned char)f;
        }
        __syncthreads();
    }
}

// g(x) = amp exp(-d^2/(2 sigma^2)), d the periodic minimum-image x - x0;
// E_z: q2 = g, q4 = -g; E_y: q1 = g, q5 = g; other components 0.
template <typename T>
__global__ void pulse_kernel(T *__restrict__ q, int Nx, int Ny, int pol, double x0, double sigma, double amp) {
    const size_t P = size_t(Nx) * size_t(Ny);
    for (size_t i = blockIdx.x * size_t(blockDim.x) + threadIdx.x; i < P; i += size_t(gridDim.x) * blockDim.x) {
        const int x = int(i % Nx);
        double d = double(x) - x0;
        d -= double(Nx) * floor(d / double(Nx) + 0.5);
        const double g = amp * exp(-d * d / (2.0 * sigma * sigma));
        T v[6] = {T(0), T(0), T(0), T(0), T(0), T(0)};
        if (pol == 0) {
            v[2] = T(g);
            v[4] = T(-g);
        } else {
            v[1] = T(g);
            v[5] = T(g);
        }
#pragma unroll
        for (int c = 0; c < 6; ++c) q[size_t(c) * P + i] = v[c];
    }
}

template <typename S, typename D>
__global__ void convert_kernel(const S *__restrict__ src, D *__restrict__ dst, size_t n) {
    for (size_t i = blockIdx.x * size_t(blockDim.x) + threadIdx.x; i < n; i += size_t(gridDim.x) * blockDim.x)
        dst[i] = D(src[i]);
}

int grid_for(size_t n, int block) {
    size_t g = (n + block - 1) / block;
    if (g > 152 * 32) g = 152 * 32;
    if (g < 1) g = 1;
    return int(g);
}

}  // namespace

namespace {
// Smallest and largest value of a plane (16 independent chains; one alone is bound
// by the latency of its comparisons).
void plane_range(const double *n, size_t P, double range[2]) {
    constexpr int L = 16;
    double lo[L], hi[L];
    for (int k = 0; k < L; ++k) lo[k] = hi[k] = n[0];
    auto take = [&](int k, double v) {
        lo[k] = v < lo[k] ? v : lo[k];
        hi[k] = v > hi[k] ? v : hi[k];
    };
    size_t i = 0;
    for (; i + L <= P; i += L)
        for (int k = 0; k < L; ++k) take(k, n[i + k]);
    for (; i < P; ++i) take(0, n[i]);
    range[0] = *std::min_element(lo, lo + L);
    range[1] = *std::max_element(hi, hi + L);
}
}  // namespace

bool index_valid(const double *n, size_t P, bool *ordinary) {
    constexpr size_t BLOCK = 1024;  // without a branch per value
    for (size_t i0 = 0; i0 < P; i0 += BLOCK) {
        const size_t i1 = std::min(P, i0 + BLOCK);
        unsigned long long outside = 0;
        for (size_t i = i0; i < i1; ++i)
            outside += 1ull - (unsigned long long)((n[i] >= kOrdinaryIndex[0]) & (n[i] <= kOrdinaryIndex[1]));
        if (outside == 0) continue;
        *ordinary = false;
        for (size_t i = i0; i < i1; ++i)
            if (!(n[i] > 0.0) || !std::isfinite(n[i])) return false;
    }
    return true;
}

int rotation_mode(const double *const n[3], bool ordinary, int Nx, int Ny, double delta, int precision, int interleaved,
                  int unitary) {
    const int mode = unitary ? MODE_UNITARY : 0;
    if (ordinary) return mode;
    if (precision == 0 && !unitary) return mode;  // collisions are shears, potential rows no rotations
    double range[3][2];
    for (int k = 0; k < 3; ++k) {
        plane_range(n[k], size_t(Nx) * Ny, range[k]);
        if (delta / (4.0 * range[k][0]) > kHalfAngleLimit) return mode | MODE_WIDE;  // Eq. 24
    }
    if (!unitary) return mode;
    // Eq. 25: n_y along x, n_x along y, n_z along both. Sites are looked at only if
    // the planes' ranges leave the possibility.
    const double scale = 0.5 * delta * (interleaved ? 0.5 : 1.0) * 0.5;
    for (int k = 0; k < 3; ++k) {
        if (scale * (range[k][1] - range[k][0]) / (range[k][0] * range[k][0]) <= kHalfAngleLimit) continue;
        const double *const p = n[k];
        for (int y = 0; y < Ny; ++y) {
            const double *const r = p + size_t(y) * Nx;
            const double *const up = p + size_t(y + 1 == Ny ? 0 : y + 1) * Nx, *const dn = p + size_t(y ? y - 1 : Ny - 1) * Nx;
            for (int x = 0; x < Nx; ++x) {
                const double dx = r[x + 1 == Nx ? 0 : x + 1] - r[x ? x - 1 : Nx - 1], dy = up[x] - dn[x];
                const double d = fmax(k != 0 ? fabs(dx) : 0.0, k != 1 ? fabs(dy) : 0.0);
                if (!(scale * d / (r[x] * r[x]) <= kHalfAngleLimit)) return mode | MODE_WIDE;
            }
        }
    }
    return mode;
}

cudaError_t launch_coefficients(const double *n, void *coef, int Nx, int Ny, double delta, int precision,
                                int interleaved, int mode, cudaStream_t st) {
    const size_t P = size_t(Nx) * size_t(Ny);
    const int B = 256;
    if (precision == 0)
        coef_kernel<float><<<grid_for(P, B), B, 0, st>>>(n, static_cast<float *>(coef), Nx, Ny, delta,
                                                          interleaved, mode);
    else
        coef_kernel<double><<<grid_for(P, B), B, 0, st>>>(n, static_cast<double *>(coef), Nx, Ny, delta,
                                                           interleaved, mode);
    return cudaGetLastError();
}

cudaError_t launch_march_records(const MarchGeo &g, const double *n, void *mem, int nfam, int fam0, double delta,
                                 int precision, int interleaved, int mode, cudaStream_t st) {
    char *m = static_cast<char *>(mem);
    const int rows = MARCH_ABOVE + g.Ny + MARCH_BELOW;
    const int fblocks = (g.Ny + FLAG_ROWS - 1) / FLAG_ROWS;
    const dim3 grid(unsigned(g.strips), unsigned(rows < 4096 ? rows : 4096));
    const dim3 fgrid(unsigned(g.strips), unsigned(fblocks < 4096 ? fblocks : 4096));
    for (int z = 0; z < nfam; ++z) {
        void *rec = m + z * g.record_bytes;
        unsigned char *flags = reinterpret_cast<unsigned char *>(m + nfam * g.record_bytes + z * g.flag_bytes);
        if (precision == 0) {
            march_records_kernel<float><<<grid, g.W, 0, st>>>(n, static_cast<float *>(rec), fam0 + z, g, delta,
                                                              interleaved, mode);
            march_flags_kernel<float><<<fgrid, 256, 0, st>>>(static_cast<const float *>(rec), flags, fam0 + z, g);
        } else {
            march_records_kernel<double><<<grid, g.W, 0, st>>>(n, static_cast<double *>(rec), fam0 + z, g, delta,
                                                               interleaved, mode);
            march_flags_kernel<double><<<fgrid, 256, 0, st>>>(static_cast<const double *>(rec), flags, fam0 + z, g);
        }
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_init_pulse(void *q, int Nx, int Ny, int precision, int pol, double x0, double sigma,
                              double amp, cudaStream_t st) {
    const size_t P = size_t(Nx) * size_t(Ny);
    const int B = 256;
    if (precision == 0)
        pulse_kernel<float><<<grid_for(P, B), B, 0, st>>>(static_cast<float *>(q), Nx, Ny, pol, x0, sigma, amp);
    else
        pulse_kernel<double><<<grid_for(P, B), B, 0, st>>>(static_cast<double *>(q), Nx, Ny, pol, x0, sigma, amp);
    return cudaGetLastError();
}

cudaError_t launch_convert(const void *src, int src_double, void *dst, int dst_double, size_t n, cudaStream_t st) {
    const int B = 256;
    const int G = grid_for(n, B);
    if (src_double && dst_double)
        convert_kernel<double, double><<<G, B, 0, st>>>(static_cast<const double *>(src), static_cast<double *>(dst), n);
    else if (src_double)
        convert_kernel<double, float><<<G, B, 0, st>>>(static_cast<const double *>(src), static_cast<float *>(dst), n);
    else if (dst_double)
        convert_kernel<float, double><<<G, B, 0, st>>>(static_cast<const float *>(src), static_cast<double *>(dst), n);
    else
        convert_kernel<float, float><<<G, B, 0, st>>>(static_cast<const float *>(src), static_cast<float *>(dst), n);
    return cudaGetLastError();
}

}  // namespace qla
