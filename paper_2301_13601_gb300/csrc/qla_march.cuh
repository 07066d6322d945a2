// Marching form of the fused sweep: K full QLA time steps per HBM pass with
// the state held in registers.
//
// The operators of a step (Eq. 18, 20, 22, 23, 28) and their per-site
// arithmetic are those of qla_sweep.cuh (rot, vop_pair; families as there), in
// the same order, so both forms give the same values. What differs is where a
// row lives between its operators:
//  * A warp owns a strip of 32 C columns (C consecutive columns per lane) and
//    marches down its rows alone. The x operators of a row act on the lane's C
//    registers (shifts are register renames plus one warp shuffle); the y
//    operators follow on the same registers, each y-shift a saved register per
//    column, the output trailing the input by 4 rows. The K time levels are
//    chained in the warp: level j's output row is level j+1's input row one
//    iteration later (one row of lag, so that the levels of an iteration do not
//    depend on each other and their operations interleave). No state passes
//    through shared memory and no block barrier is needed.
//  * The strip carries a halo of at least 4K columns on each side; the columns
//    between are written. A share of rows [y0, y1) is fed from y0 - 4K.
//  * FP32 arithmetic is packed: two of a lane's columns per fma.rn.f32x2 (the
//    same roundings as two scalar FMAs). Measured on GB300 with independent
//    rotations in registers: 28 T FMA/s scalar, 36 packed, in half the issue
//    slots.
//  * Input rows (three state planes and the collision coefficients of level 0)
//    are copied by cp.async into a ring of D rows private to the warp, D - 1
//    rows ahead; the collision coefficients of the later levels, which the L2
//    still holds, one row ahead. Every lane copies exactly what it reads.
//  * V_X' and V_Y' are the identity where their angles vanish. A flag per strip
//    and row (launch_march_records) says whether any angle is nonzero in the
//    rows that a group of iterations starting there applies; groups without one
//    neither load the V planes nor apply them.
//  * A second flag says whether the collision coefficients change from row to
//    row anywhere near the group. Where they do not (a uniform medium, or one
//    layered along x), the ring slots already hold what a copy would bring, and
//    none is issued: 66 instead of 88 bytes of DRAM traffic per site and pass at
//    8192^2 (a uniform medium around one object), 20 time steps 9.98 -> 9.67 ms.
// Coefficients lie in records, one per strip and row: MARCH_FIELDS rows of the
// strip's 32 C columns (halo included), periodic rows repeated above and below,
// so that every coefficient copy of an iteration, whatever its level and lag, is
// one address register plus a constant, aligned for any Nx.
// Measured on GB300 against the shared-memory sweep (us per step, both families,
// interleaved with other contexts' calls): 8192^2 810 -> 480 (140 G site-updates/s,
// 3.5 TB/s of HBM traffic), 2048^2 78 -> 39, 1024^2 44 -> 13, 256^2 26 -> 4; 4096^2,
// one family, 106 -> 65; 256^2 FP64 330 -> 62. That sweep was bound by instruction
// issue (half of its instructions index and control work) and its two block
// barriers per row block; this one by the fixed latencies of its chains with the 8
// warps per SM that 247 registers leave (two steps; issue slots 41% busy, FMA pipe
// 38%), on the smallest lattices by the latency of a pass. On the way there
// (8192^2): one body per family and with and without potentials, scalar FMAs 925 us
// (instruction cache); one body for both families 731; packed FMAs 628; planes by
// 32-bit offsets 591; coefficient records 538; row ranges by measured costs 505.
#pragma once

#include "qla_sweep.cuh"

namespace qla {

constexpr int MARCH_LAG = 1;    // rows between a level's output and the next level's input

// Iterations of a share before its first output row leaves: level j works on
// row F0 + it - (4 + MARCH_LAG) j in iteration it, F0 = y0 - 4K.
constexpr int march_delay(int K) { return 8 * K + MARCH_LAG * (K - 1); }
static_assert(march_flag_back(2) >= (4 + MARCH_LAG) + 4, "V rows of a group");

// A family's planes and what distinguishes the families at run time (one code
// serves both, so that the warps of an SM share its instruction cache whatever
// their family). The TE hub is carried with its sign flipped, which turns the
// orientations of all of its operators into the TM ones (IEEE arithmetic is
// symmetric under it, so the values are unchanged); what remains is which
// member the printed potential rows write.
struct MarchFam {
    const char *h, *px, *py;        // input planes
    const char *rec;                // coefficient records
    char *oh, *opx, *opy;           // output planes
    const unsigned char *flags;     // [strips][Ny]
    int te;
};

struct MarchArgs {
    MarchFam fam[2];  // the advanced families, in grid order
    int Nx, Ny;
    int w_valid, halo, strips;  // strip geometry (MarchGeo)
    int chunks;                 // row ranges per strip, one warp each
    int ctas_fam;               // CTAs per family
    int chained;                // the launch before it on the stream is a pass over the same records
};

template <typename T, int C, int K, int D, bool INTER>
struct MarchLayout {
    static_assert(D == 2 || D == 3, "copy groups in flight");
    static constexpr int W = 32 * C;
    static constexpr int RB = W * int(sizeof(T));  // one row of a plane
    static constexpr int REC = 7 * RB;             // a level-0 row: h, x-partner, y-partner, C_X (2), C_Y (2)
    static constexpr int CREC = 4 * RB;            // a later level's C_X, C_Y
    static constexpr int VYS = INTER ? 4 : 2;      // rows of V_Y kept (Eq. 28 applies it at lags 2 and 4)
    static constexpr int VREC = (2 + VYS) * 2 * RB;  // per level: V_X (two rows), V_Y
    static constexpr int C_OFF = D * REC;
    static constexpr int V_OFF = C_OFF + (K - 1) * 2 * CREC;
    static constexpr int WARP = V_OFF + K * VREC;
};

// ---- vectors of a lane's columns --------------------------------------------
// FP32: packed pairs; FP64: scalars. NV vectors hold the lane's C columns.
struct F32x2 {
    unsigned long long v;
};
template <typename T>
struct MarchVec;
template <>
struct MarchVec<float> {
    using V = F32x2;
    static constexpr int N = 2;
    static __device__ __forceinline__ V pack(float a, float b) {
        V r;
        asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
        return r;
    }
    static __device__ __forceinline__ void unpack(V v, float &a, float &b) {
        asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v.v));
    }
    static __device__ __forceinline__ V neg(V a) {
        float x, y;
        unpack(a, x, y);
        return pack(-x, -y);
    }
    static __device__ __forceinline__ V fma(V a, V b, V c) {
        V r;
        asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
        return r;
    }
    static __device__ __forceinline__ V mul(V a, V b) {
        V r;
        asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
        return r;
    }
    static __device__ __forceinline__ V add(V a, V b) {
        V r;
        asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
        return r;
    }
    static __device__ __forceinline__ V zero() { return V{0ull}; }
    static __device__ __forceinline__ V flip(V a, unsigned mask) {
        return V{a.v ^ ((unsigned long long)(mask) << 32 | mask)};
    }
};
template <>
struct MarchVec<double> {
    using V = double;
    static constexpr int N = 1;
    static __device__ __forceinline__ V neg(V a) { return -a; }
    static __device__ __forceinline__ V fma(V a, V b, V c) { return __fma_rn(a, b, c); }
    static __device__ __forceinline__ V mul(V a, V b) { return __dmul_rn(a, b); }
    static __device__ __forceinline__ V add(V a, V b) { return __dadd_rn(a, b); }
    static __device__ __forceinline__ V zero() { return 0.0; }
    static __device__ __forceinline__ V flip(V a, unsigned mask) {
        return __hiloint2double(__double2hiint(a) ^ int(mask), __double2loint(a));
    }
};

// rot and vop_pair of qla_sweep.cuh on vectors.
template <bool DAG, int SG, RotForm FORM, typename T, typename V = typename MarchVec<T>::V>
__device__ __forceinline__ void march_rot(V &h, V &p, V m, V s) {
    using A = MarchVec<T>;
    constexpr bool pos = (SG > 0) != DAG;
    if constexpr (FORM == ROT_SHEAR) {
        h = A::fma(pos ? m : A::neg(m), p, h);
        p = A::fma(pos ? A::neg(s) : s, h, p);
        h = A::fma(pos ? m : A::neg(m), p, h);
    } else if constexpr (FORM == ROT_WIDE) {
        const V sp = A::mul(s, p), sh = A::mul(s, h);
        const V u = A::fma(m, h, pos ? sp : A::neg(sp)), v = A::fma(m, p, pos ? A::neg(sh) : sh);
        h = A::add(h, u);
        p = A::add(p, v);
    } else {
        const V t = pos ? A::neg(m) : m, u = A::fma(t, h, p);
        if constexpr (sizeof(T) == 4) {
            const V h0 = h;
            h = A::fma(pos ? s : A::neg(s), u, h);
            p = A::fma(t, A::add(h0, h), p);
        } else {
            const V v = A::fma(A::neg(t), p, h);
            h = A::fma(pos ? s : A::neg(s), u, h);
            p = A::fma(pos ? A::neg(s) : s, v, p);
        }
    }
}
template <int TAU, bool HUB, int MODE, typename T, typename V = typename MarchVec<T>::V>
__device__ __forceinline__ void march_vop(V &h, V &p, V s, V c) {
    using A = MarchVec<T>;
    V &t = HUB ? h : p;
    V &src = HUB ? p : h;
    if constexpr (MODE & MODE_UNITARY) {
        march_rot<false, TAU, rot_form<T, MODE>(), T>(t, src, c, s);
    } else {
        const V ss = A::mul(s, src);
        t = A::add(t, A::fma(c, t, TAU > 0 ? ss : A::neg(ss)));
    }
}

// A lane's vectors. FP64: its columns in order. FP32: columns (0, 2) and (1, 3) of
// its four (march_column), so that a shift by one column is a rename, one shuffle
// and one register move: of pairs (0, 1), (2, 3) it takes three moves (2048^2 39.8
// -> 38.5 us per step, unitary 1536 x 1000 18.7 -> 17.2). Records hold the columns
// in that order; state rows are regrouped where a lane reads and writes them.
//
// a(x) <- a(x-1), a(x) <- a(x+1) across the warp's 32 C columns
template <typename T, int NV, typename V = typename MarchVec<T>::V>
__device__ __forceinline__ void march_from_left(V (&a)[NV]) {
    if constexpr (MarchVec<T>::N == 2) {
        static_assert(NV == 2, "four columns");
        float x1, x3;
        MarchVec<T>::unpack(a[1], x1, x3);
        const float e = __shfl_up_sync(0xffffffffu, x3, 1);
        a[1] = a[0];
        a[0] = MarchVec<T>::pack(e, x1);
    } else {
        const V e = __shfl_up_sync(0xffffffffu, a[NV - 1], 1);
#pragma unroll
        for (int k = NV - 1; k > 0; --k) a[k] = a[k - 1];
        a[0] = e;
    }
}
template <typename T, int NV, typename V = typename MarchVec<T>::V>
__device__ __forceinline__ void march_from_right(V (&a)[NV]) {
    if constexpr (MarchVec<T>::N == 2) {
        static_assert(NV == 2, "four columns");
        float x0, x2;
        MarchVec<T>::unpack(a[0], x0, x2);
        const float e = __shfl_down_sync(0xffffffffu, x0, 1);
        a[0] = a[1];
        a[1] = MarchVec<T>::pack(x2, e);
    } else {
        const V e = __shfl_down_sync(0xffffffffu, a[0], 1);
#pragma unroll
        for (int k = 0; k + 1 < NV; ++k) a[k] = a[k + 1];
        a[NV - 1] = e;
    }
}

// The lane's NV vectors of a staged record row, whose values lie in the order of
// the vectors (p: its first byte); of a staged state row; and their store.
template <typename T, int NV, typename V = typename MarchVec<T>::V>
__device__ __forceinline__ void march_lds(V (&v)[NV], const unsigned char *p) {
    static_assert(sizeof(V) * NV == 16, "16 bytes per lane");
    const ulonglong2 a = *reinterpret_cast<const ulonglong2 *>(p);
    memcpy(&v[0], &a.x, 8);
    memcpy(&v[1], &a.y, 8);
}
template <typename T, int NV, typename V = typename MarchVec<T>::V>
__device__ __forceinline__ void march_lds_state(V (&v)[NV], const unsigned char *p) {
    if constexpr (MarchVec<T>::N == 2) {
        const float4 a = *reinterpret_cast<const float4 *>(p);
        v[0] = MarchVec<T>::pack(a.x, a.z);
        v[1] = MarchVec<T>::pack(a.y, a.w);
    } else {
        march_lds<T, NV>(v, p);
    }
}
template <typename T, int C, int NV, typename V = typename MarchVec<T>::V>
__device__ __forceinline__ void march_columns(T (&x)[C], const V (&v)[NV]) {
    if constexpr (MarchVec<T>::N == 2) {
        MarchVec<T>::unpack(v[0], x[0], x[2]);
        MarchVec<T>::unpack(v[1], x[1], x[3]);
    } else {
#pragma unroll
        for (int k = 0; k < C; ++k) x[k] = v[k];
    }
}
template <typename T, int C, int NV, typename V = typename MarchVec<T>::V>
__device__ __forceinline__ void march_stg(T *dst, const V (&v)[NV]) {
    T x[C];
    march_columns<T, C, NV>(x, v);
    if constexpr (C == 4)
        *reinterpret_cast<float4 *>(dst) = make_float4(x[0], x[1], x[2], x[3]);
    else
        *reinterpret_cast<double2 *>(dst) = make_double2(x[0], x[1]);
}
template <typename T, int C, int NV, typename V = typename MarchVec<T>::V>
__device__ __forceinline__ void march_stg_some(T *dst, const V (&v)[NV], const bool (&ok)[C]) {
    T x[C];
    march_columns<T, C, NV>(x, v);
#pragma unroll
    for (int k = 0; k < C; ++k)
        if (ok[k]) dst[k] = x[k];
}

template <int BYTES>
__device__ __forceinline__ void march_cp(unsigned dst, const void *src) {
    if constexpr (BYTES == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(src) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(dst), "l"(src), "n"(BYTES) : "memory");
}

// One time level's y pipeline: a saved value per y-shift, the collision
// coefficients of the last three rows and the x-partner's last four rows.
template <typename V, int NV>
struct MarchPipe {
    V S[8][NV];
    V m[3][NV], s[3][NV];
    V d[4][NV];
};

static_assert(Fam<1>::SGX == -Fam<0>::SGX && Fam<1>::SGY == -Fam<0>::SGY && Fam<1>::TX == -Fam<0>::TX &&
                  Fam<1>::TY == -Fam<0>::TY,
              "a sign flip of the hub maps the TE orientations to the TM ones");
static_assert(!Fam<0>::VX_HUB && !Fam<0>::VY_HUB && Fam<1>::VX_HUB && Fam<1>::VY_HUB, "potential targets");

// V' on the lane's columns of all levels (ld loads level j's coefficients).
template <int TAU, int MODE, typename T, int K, int NV, typename V, class LD>
__device__ __forceinline__ void march_v(bool te, V (&h)[K][NV], V (&p)[K][NV], LD &&ld) {
#pragma unroll
    for (int j = 0; j < K; ++j) {
        V m[NV], s[NV];
        ld(j, m, s);
        if (te) {
#pragma unroll
            for (int c = 0; c < NV; ++c) march_vop<TAU, true, MODE, T>(h[j][c], p[j][c], s[c], m[c]);
        } else {
#pragma unroll
            for (int c = 0; c < NV; ++c) march_vop<TAU, false, MODE, T>(h[j][c], p[j][c], s[c], m[c]);
        }
    }
}

// One row of every level: level j's h, p (y-partner), px (x-partner) enter as
// row R_j of its input and leave as row R_j - 4 of its output. vx, vy2, vy4
// load the V coefficients (V_X of row R, or of R - 4 with Eq. 23; V_Y of rows
// R - 2 and R - 4).
template <bool INTER, int MODE, typename T, int K, int NV, typename V, class VX, class VY2, class VY4>
__device__ __forceinline__ void march_rows(MarchPipe<V, NV> (&Y)[K], V (&h)[K][NV], V (&p)[K][NV], V (&px)[K][NV],
                                           const V (&cxm)[K][NV], const V (&cxs)[K][NV], const V (&cym)[K][NV],
                                           const V (&cys)[K][NV], bool von, bool te, VX &&vx, VY2 &&vy2, VY4 &&vy4) {
    using Fm = Fam<0>;
    constexpr RotForm SHR = rot_form<T, MODE>();
    constexpr int SX = Fm::SGX, SY = Fm::SGY;
#define MARCH_ALL(expr)               \
    _Pragma("unroll") for (int j = 0; j < K; ++j) { expr; }
#define MARCH_ROT(DAG, SG, H, PP, M, S) \
    _Pragma("unroll") for (int j = 0; j < K; ++j) _Pragma("unroll") for (int c = 0; c < NV; ++c) \
        march_rot<DAG, SG, SHR, T>(H[j][c], PP[j][c], M[c], S[c]);
#define MARCH_X(DAG) MARCH_ROT(DAG, SX, h, px, cxm[j], cxs[j])
#define MARCH_Y(DAG, M, S) MARCH_ROT(DAG, SY, h, p, M, S)
    MARCH_X(true)
    MARCH_ALL((march_from_left<T, NV>(px[j])))
    MARCH_X(false)
    MARCH_ALL((march_from_right<T, NV>(px[j])))
    MARCH_X(true)
    MARCH_ALL((march_from_right<T, NV>(h[j])))
    MARCH_X(false)
    MARCH_ALL((march_from_left<T, NV>(h[j])))
    if constexpr (INTER) {
        if (von) march_v<Fm::TX, MODE, T, K, NV, V>(te, h, px, vx);
    }
    MARCH_X(false)
    MARCH_ALL((march_from_right<T, NV>(px[j])))
    MARCH_X(true)
    MARCH_ALL((march_from_left<T, NV>(px[j])))
    MARCH_X(false)
    MARCH_ALL((march_from_left<T, NV>(h[j])))
    MARCH_X(true)
    MARCH_ALL((march_from_right<T, NV>(h[j])))
    if constexpr (INTER) {
        if (von) march_v<Fm::TX, MODE, T, K, NV, V>(te, h, px, vx);
    }
    auto swap = [&](V (&a)[NV], V (&b)[NV]) {
#pragma unroll
        for (int c = 0; c < NV; ++c) {
            const V t = a[c];
            a[c] = b[c];
            b[c] = t;
        }
    };
    MARCH_Y(true, cym[j], cys[j])         // C+   (row R)
    MARCH_ALL(swap(Y[j].S[0], p[j]))      // p <- p(r-1)
    MARCH_Y(false, cym[j], cys[j])        // C    (row R)
    MARCH_ALL(swap(Y[j].S[1], h[j]))      // p <- p(r+1): now row R-1
    MARCH_Y(true, Y[j].m[0], Y[j].s[0])   // C+   (row R-1)
    MARCH_ALL(swap(Y[j].S[2], p[j]))      // h <- h(r+1): now row R-2
    MARCH_Y(false, Y[j].m[1], Y[j].s[1])  // C    (row R-2)
    MARCH_ALL(swap(Y[j].S[3], h[j]))      // h <- h(r-1)
    if constexpr (INTER) {
        if (von) march_v<Fm::TY, MODE, T, K, NV, V>(te, h, p, vy2);  // V_Y' (row R-2)
    }
    MARCH_Y(false, Y[j].m[1], Y[j].s[1])  // C    (row R-2)
    MARCH_ALL(swap(Y[j].S[4], h[j]))      // p <- p(r+1): now row R-3
    MARCH_Y(true, Y[j].m[2], Y[j].s[2])   // C+   (row R-3)
    MARCH_ALL(swap(Y[j].S[5], p[j]))      // p <- p(r-1)
    MARCH_Y(false, Y[j].m[2], Y[j].s[2])  // C    (row R-3)
    MARCH_ALL(swap(Y[j].S[6], h[j]))      // h <- h(r-1)
    MARCH_Y(true, Y[j].m[2], Y[j].s[2])   // C+   (row R-3)
    MARCH_ALL(swap(Y[j].S[7], p[j]))      // h <- h(r+1): now row R-4
#pragma unroll
    for (int j = 0; j < K; ++j)
#pragma unroll
        for (int c = 0; c < NV; ++c) {
            const V t = Y[j].d[3][c];  // the x-partner's row R-4
            Y[j].d[3][c] = Y[j].d[2][c];
            Y[j].d[2][c] = Y[j].d[1][c];
            Y[j].d[1][c] = Y[j].d[0][c];
            Y[j].d[0][c] = px[j][c];
            px[j][c] = t;
            Y[j].m[2][c] = Y[j].m[1][c];
            Y[j].s[2][c] = Y[j].s[1][c];
            Y[j].m[1][c] = Y[j].m[0][c];
            Y[j].s[1][c] = Y[j].s[0][c];
            Y[j].m[0][c] = cym[j][c];
            Y[j].s[0][c] = cys[j][c];
        }
    if (von) {
        if constexpr (!INTER) march_v<Fm::TX, MODE, T, K, NV, V>(te, h, px, vx);  // V_X (row R-4)
        march_v<Fm::TY, MODE, T, K, NV, V>(te, h, p, vy4);                        // V_Y (row R-4)
    }
#undef MARCH_ALL
#undef MARCH_ROT
#undef MARCH_X
#undef MARCH_Y
}

// One warp's share: rows [y0, y1) of strip `strip` of a family. sm: the
// warp's shared memory. VEC: rows keep the alignment of the lane's vectors (Nx a
// multiple of C) and a plane holds less than 2^32 bytes; else the state is copied
// and stored element by element, with 64-bit offsets.
// Passes of one FP32 step are chained: each may be launched while the one before
// it finishes its last group of rows, and waits for its end before it reads the
// state (griddepcontrol). Such a pass, on a small lattice, is about as long as a
// launch takes: 16 steps of 256^2 76 -> 64 us. Passes of two FP32 steps are not:
// they are longer, and the two instructions cost the fullest register file 3%
// (2048^2 4.02 -> 4.14 ms, 8192^2 9.85 -> 10.15); nor are FP64's, whose waiting
// CTAs keep other streams' CTAs off the pipe (256^2 1.23 -> 1.26 ms).
template <typename T>
constexpr bool march_chains(int K) {
    return sizeof(T) == 4 && K == 1;
}

template <typename T, int C, int K, int D, int U, bool INTER, int MODE, bool VEC, bool CHAIN>
__device__ __forceinline__ void march_share(const MarchArgs &A, const MarchFam &F, int strip, int y0, int y1, unsigned char *sm,
                                            int lane) {
    using L = MarchLayout<T, C, K, D, INTER>;
    using MV = MarchVec<T>;
    using V = typename MV::V;
    constexpr int NV = C / MV::N;
    static_assert(NV * MV::N == C, "whole vectors");
    constexpr int LB = C * int(sizeof(T));  // a lane's bytes of a row
    constexpr int RB = L::RB;
    const int Nx = A.Nx, Ny = A.Ny;
    // Places in a plane as byte offsets from plane addresses that lie in the
    // kernel's parameters; 32-bit ones (VEC) take one register and little
    // arithmetic (8192^2: 628 -> 591 us per step).
    using Off = std::conditional_t<VEC, unsigned, size_t>;
    const Off pitch = Off(Nx) * Off(sizeof(T)), plane_bytes = pitch * Off(Ny);
    const bool te = F.te != 0;
    const unsigned hsign = te ? 0x80000000u : 0u;
    const int cy_off = te ? 2 * RB : 0;  // TM: C_X and C_Y are one plane

    const int o_lo = strip * A.w_valid;
    const int o_hi = min(o_lo + A.w_valid, Nx);
    const int xbase = o_lo - A.halo;
    constexpr int NGC = VEC ? 1 : C;  // global columns of the lane (VEC: of its first column)
    Off gc[NGC];
#pragma unroll
    for (int k = 0; k < NGC; ++k) gc[k] = Off(wrapi(xbase + C * lane + k, Nx)) * Off(sizeof(T));
    const unsigned sbase = tc::smem_addr(sm) + unsigned(lane) * LB;
    sm += lane * LB;

    const int F0 = y0 - 4 * K;
    // ro: byte offset of the row (VEC: of the lane's first column in it)
    auto row = [&](unsigned dst, const char *plane, Off ro) {
        if constexpr (VEC) {
            march_cp<LB>(dst, plane + ro);
        } else {
#pragma unroll
            for (int k = 0; k < C; ++k) march_cp<sizeof(T)>(dst + k * unsigned(sizeof(T)), plane + ro + gc[k]);
        }
    };
    // coefficient copies: two fields (x, y) of the record `dr` rows from the
    // level-0 row that cp points to
    constexpr int RECB = MARCH_FIELDS * RB;
    const char *cp = F.rec + (size_t(strip) * (MARCH_ABOVE + Ny + MARCH_BELOW) + size_t(MARCH_ABOVE + F0)) * RECB +
                     lane * LB;
    auto field2 = [&](unsigned dst, int dr, int field) {
        march_cp<LB>(dst, cp + (dr * RECB + field * RB));
        march_cp<LB>(dst + RB, cp + (dr * RECB + (field + 1) * RB));
    };
    auto copy0 = [&](unsigned slot_off, Off ro, int dr, bool coefs) {
        const unsigned b = sbase + slot_off;
        row(b, F.h, ro);
        row(b + RB, F.px, ro);
        row(b + 2 * RB, F.py, ro);
        if (coefs) {
            field2(b + 3 * RB, dr, F_CX);
            if (te) field2(b + 5 * RB, dr, F_CY);
        }
    };
    auto copyc = [&](int j, int slot, int dr) {
        const unsigned b = sbase + L::C_OFF + ((j - 1) * 2 + slot) * L::CREC;
        field2(b, dr, F_CX);
        if (te) field2(b + 2 * RB, dr, F_CY);
    };
    // V rows that level j applies in iteration i (dr: its level row from cp)
    auto copyv = [&](int j, int i, int dr) {
        const unsigned b = sbase + L::V_OFF + j * L::VREC;
        if constexpr (INTER) {
            field2(b + (i & 1) * 2 * RB, dr, F_VX);
            field2(b + (2 + ((i + 2) & 3)) * 2 * RB, dr - 2, F_VY);
        } else {
            field2(b + (i & 1) * 2 * RB, dr - 4, F_VX);
            field2(b + (2 + (i & 1)) * 2 * RB, dr - 4, F_VY);
        }
    };

    MarchPipe<V, NV> pipe[K];
    V hh[K][NV], hp[K][NV], hx[K][NV];  // the rows entering each level (level 0: from the ring)
#pragma unroll
    for (int j = 0; j < K; ++j)
#pragma unroll
        for (int c = 0; c < NV; ++c) {
#pragma unroll
            for (int k = 0; k < 8; ++k) pipe[j].S[k][c] = MV::zero();
#pragma unroll
            for (int k = 0; k < 3; ++k) pipe[j].m[k][c] = pipe[j].s[k][c] = MV::zero();
#pragma unroll
            for (int k = 0; k < 4; ++k) pipe[j].d[k][c] = MV::zero();
            hh[j][c] = hp[j][c] = hx[j][c] = MV::zero();
        }

    const unsigned char *const flags = F.flags + size_t(strip) * Ny;
    const int nit = y1 - y0 + march_delay(K);
    const int ngroups = (nit + U - 1) / U;
    int rg = wrapi(F0, Ny);  // wrapped level-0 row of the group's first iteration
    auto step_row = [&](int &r, Off &off) {  // next row, wrapped (r counts up to 0 at the wrap)
        off += pitch;
        if (++r == 0) {
            r = -Ny;
            off -= plane_bytes;
        }
    };
    // prologue: level-0 rows F0 .. F0 + D - 2, the later levels' first collision rows, the first V rows
    unsigned von = flags[rg], von1 = flags[wrapi(rg + U, Ny)], von2 = flags[wrapi(rg + 2 * U, Ny)];
    int row_c = rg - Ny;  // level-0 copies
    Off off_c = Off(rg) * pitch + (VEC ? gc[0] : Off(0));
#pragma unroll
    for (int j = 1; j < K; ++j) copyc(j, 0, -(4 + MARCH_LAG) * j);
    if (von & MARCH_V)
        for (int j = 0; j < K; ++j) copyv(j, 0, -(4 + MARCH_LAG) * j);
    if constexpr (CHAIN) asm volatile("griddepcontrol.wait;\n" ::: "memory");
#pragma unroll
    for (int k = 0; k < D - 1; ++k) {
        copy0(k * L::REC, off_c, k, true);
        step_row(row_c, off_c);
        cp_async_commit();
    }
    unsigned rd_off = 0, wr_off = (D - 1) * L::REC;

    // output: row y0 + it - march_delay(K)
    bool ok[NGC];
#pragma unroll
    for (int k = 0; k < NGC; ++k) {
        const int c = C * lane + k;
        ok[k] = c >= A.halo && xbase + c < o_hi;
    }
    const int n_out = y1 - y0;
    // (offsets of rows and columns that are not written wrap around harmlessly)
    Off out_off = Off(y0 - march_delay(K)) * pitch + Off(xbase + C * lane) * Off(sizeof(T));

    for (int g = 0, it0 = 0; g < ngroups; ++g, it0 += U) {
        const unsigned von3 = flags[wrap_down(rg + 3 * U, Ny)];  // read three groups ahead
        // V_Y rows are copied up to four iterations before their last use
        const bool on = (von & MARCH_V) != 0, vcopy = ((von | von1 | (U < 4 ? von2 : 0u)) & MARCH_V) != 0;
        // (the first D - 1 rows came with the prologue, the ring is full after iteration 0)
        const bool ccopy = it0 == 0 || (von & MARCH_C) != 0;
        if constexpr (CHAIN)
            if (g == ngroups - 1) asm volatile("griddepcontrol.launch_dependents;\n");
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int i = U == 4 ? u : it0 + u;  // iteration index mod 4 (compile time when U = 4)
            // all copies but the newest level-0 row's have landed (a lane reads only what it copied)
            asm volatile("cp.async.wait_group %0;\n" ::"n"(D - 2) : "memory");
            if (ccopy) {
#pragma unroll
                for (int j = 1; j < K; ++j) copyc(j, (i + 1) & 1, 1 - (4 + MARCH_LAG) * j);
            }
            if (vcopy) {
#pragma unroll
                for (int j = 0; j < K; ++j) copyv(j, i + 1, 1 - (4 + MARCH_LAG) * j);
            }
            if constexpr (D > 2) cp_async_commit();
            copy0(wr_off, off_c, D - 1, ccopy);
            step_row(row_c, off_c);
            cp_async_commit();
            cp += RECB;
            wr_off = wr_off == (D - 1) * L::REC ? 0u : wr_off + L::REC;

            V cxm[K][NV], cxs[K][NV], cym[K][NV], cys[K][NV];
#pragma unroll
            for (int j = 0; j < K; ++j) {
                const unsigned char *cb = sm + L::C_OFF + ((j - 1) * 2 + (i & 1)) * L::CREC;
                if (j == 0) {
                    const unsigned char *rec = sm + rd_off;
                    march_lds_state<T, NV>(hh[0], rec);
                    march_lds_state<T, NV>(hx[0], rec + RB);
                    march_lds_state<T, NV>(hp[0], rec + 2 * RB);
#pragma unroll
                    for (int c = 0; c < NV; ++c) hh[0][c] = MV::flip(hh[0][c], hsign);
                    cb = rec + 3 * RB;
                }
                march_lds<T, NV>(cxm[j], cb);
                march_lds<T, NV>(cxs[j], cb + RB);
                march_lds<T, NV>(cym[j], cb + cy_off);
                march_lds<T, NV>(cys[j], cb + cy_off + RB);
            }
            rd_off = rd_off == (D - 1) * L::REC ? 0u : rd_off + L::REC;
            auto vrow = [&](int slot) {
                return [&, slot](int j, V(&m)[NV], V(&s)[NV]) {
                    const unsigned char *vb = sm + L::V_OFF + j * L::VREC + slot * 2 * RB;
                    march_lds<T, NV>(m, vb);
                    march_lds<T, NV>(s, vb + RB);
                };
            };
            march_rows<INTER, MODE, T, K, NV, V>(pipe, hh, hp, hx, cxm, cxs, cym, cys, on, te, vrow(i & 1),
                                                 vrow(2 + ((i + 2) & 3)), vrow(INTER ? 2 + (i & 3) : 2 + (i & 1)));
            const int ro = it0 + u - march_delay(K);
            if (ro >= 0 && ro < n_out) {
                V h[NV];
#pragma unroll
                for (int c = 0; c < NV; ++c) h[c] = MV::flip(hh[K - 1][c], hsign);
                T *const oh = reinterpret_cast<T *>(F.oh + out_off), *const ox = reinterpret_cast<T *>(F.opx + out_off),
                         *const oy = reinterpret_cast<T *>(F.opy + out_off);
                if constexpr (VEC) {
                    if (ok[0]) {
                        march_stg<T, C, NV>(oh, h);
                        march_stg<T, C, NV>(ox, hx[K - 1]);
                        march_stg<T, C, NV>(oy, hp[K - 1]);
                    }
                } else {
                    march_stg_some<T, C, NV>(oh, h, ok);
                    march_stg_some<T, C, NV>(ox, hx[K - 1], ok);
                    march_stg_some<T, C, NV>(oy, hp[K - 1], ok);
                }
            }
            out_off += pitch;
#pragma unroll
            for (int j = K - 1; j > 0; --j)
#pragma unroll
                for (int c = 0; c < NV; ++c) {
                    hh[j][c] = hh[j - 1][c];
                    hp[j][c] = hp[j - 1][c];
                    hx[j][c] = hx[j - 1][c];
                }
        }
        von = von1;
        von1 = von2;
        von2 = von3;
        rg = wrap_down(rg + U, Ny);
    }
    cp_async_wait_all();
}

template <typename T, int C, int K, int D, int U, int WPC, int MINB, bool INTER, int MODE, bool VEC>
__global__ void __launch_bounds__(32 * WPC, MINB) march_kernel(const __grid_constant__ MarchArgs A) {
    using L = MarchLayout<T, C, K, D, INTER>;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31;
    const int warp = __shfl_sync(0xffffffffu, int(threadIdx.x) >> 5, 0);
    const int layer = int(blockIdx.x) >= A.ctas_fam ? 1 : 0;
    const int w = (int(blockIdx.x) - layer * A.ctas_fam) * WPC + warp;
    if (w >= A.strips * A.chunks) return;
    const int strip = w % A.strips, chunk = w / A.strips;
    const int y0 = int((long long)A.Ny * chunk / A.chunks);
    const int y1 = int((long long)A.Ny * (chunk + 1) / A.chunks);
    march_share<T, C, K, D, U, INTER, MODE, VEC, march_chains<T>(K)>(A, A.fam[layer], strip, y0, y1,
                                                                     smem_raw + warp * L::WARP, lane);
}

// A family's entry (fam: 0 = TM, 1 = TE).
template <typename T>
__host__ __device__ MarchFam march_fam(const void *q_in, void *q_out, const void *rec, const unsigned char *flags, int fam, int Nx,
                          int Ny) {
    const size_t PB = size_t(Nx) * Ny * sizeof(T);
    const char *q = static_cast<const char *>(q_in);
    char *o = static_cast<char *>(q_out);
    MarchFam f;
    const bool te = fam != 0;
    const int h = te ? Fam<1>::H : Fam<0>::H, px = te ? Fam<1>::PX : Fam<0>::PX, py = te ? Fam<1>::PY : Fam<0>::PY;
    f.h = q + h * PB;
    f.px = q + px * PB;
    f.py = q + py * PB;
    f.oh = o + h * PB;
    f.opx = o + px * PB;
    f.opy = o + py * PB;
    f.rec = static_cast<const char *>(rec);
    f.flags = flags;
    f.te = te ? 1 : 0;
    return f;
}

template <typename T, int C, int K, int D, int U, int WPC, int MINB, bool INTER, int MODE, bool VEC>
cudaError_t launch_march_t(const MarchArgs &a, int nfam, cudaStream_t st) {
    using L = MarchLayout<T, C, K, D, INTER>;
    auto kern = march_kernel<T, C, K, D, U, WPC, MINB, INTER, MODE, VEC>;
    // set on every launch: the attribute belongs to the device, a process may use several
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, L::WARP * WPC);
    if (e != cudaSuccess) return e;
    MarchArgs m = a;
    m.ctas_fam = (a.strips * a.chunks + WPC - 1) / WPC;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(unsigned(m.ctas_fam) * unsigned(nfam));
    cfg.blockDim = dim3(32 * WPC);
    cfg.dynamicSmemBytes = L::WARP * WPC;
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = march_chains<T>(K) && a.chained ? 1 : 0;
    cudaLaunchKernelEx(&cfg, kern, m);
    return cudaGetLastError();
}
template <typename T, int C, int K, int D, int U, int WPC, int MINB, bool VEC, bool INTER>
cudaError_t launch_march_mode(const MarchArgs &a, int nfam, int mode, cudaStream_t st) {
    constexpr int UW = MODE_UNITARY | MODE_WIDE;
    switch (mode) {
        case 0: return launch_march_t<T, C, K, D, U, WPC, MINB, INTER, 0, VEC>(a, nfam, st);
        case MODE_UNITARY: return launch_march_t<T, C, K, D, U, WPC, MINB, INTER, MODE_UNITARY, VEC>(a, nfam, st);
        case UW: return launch_march_t<T, C, K, D, U, WPC, MINB, INTER, UW, VEC>(a, nfam, st);
        case MODE_WIDE:  // FP32 collisions are shears then (rotation_mode)
            if constexpr (sizeof(T) == 8)
                return launch_march_t<T, C, K, D, U, WPC, MINB, INTER, MODE_WIDE, VEC>(a, nfam, st);
    }
    return cudaErrorInvalidValue;
}
template <typename T, int C, int K, int D, int U, int WPC, int MINB, bool VEC>
cudaError_t launch_march_modes(const MarchArgs &a, int nfam, int interleaved, int mode, cudaStream_t st) {
    return interleaved ? launch_march_mode<T, C, K, D, U, WPC, MINB, VEC, true>(a, nfam, mode, st)
                       : launch_march_mode<T, C, K, D, U, WPC, MINB, VEC, false>(a, nfam, mode, st);
}

// The instantiated forms, one translation unit each (qla_march_*.cu).
cudaError_t launch_march_f32_k1(const MarchArgs &a, int nfam, int interleaved, int mode, cudaStream_t st);
cudaError_t launch_march_f32_k1_any(const MarchArgs &a, int nfam, int interleaved, int mode, cudaStream_t st);
cudaError_t launch_march_f32_k2(const MarchArgs &a, int nfam, int interleaved, int mode, cudaStream_t st);
cudaError_t launch_march_f32_k2_any(const MarchArgs &a, int nfam, int interleaved, int mode, cudaStream_t st);
cudaError_t launch_march_f64_k1(const MarchArgs &a, int nfam, int interleaved, int mode, cudaStream_t st);
cudaError_t launch_march_f64_k1_any(const MarchArgs &a, int nfam, int interleaved, int mode, cudaStream_t st);

}  // namespace qla
