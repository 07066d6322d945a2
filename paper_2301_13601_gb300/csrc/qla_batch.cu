// Batched QLA: many independent lattices (of uneven sizes) advanced by one
// persistent kernel, replayed as a CUDA graph.
//
// Work items are (instance, pass of two steps, family, tile) with a tile the
// shares of four warps of the marching sweep (qla_march.cuh). Items are numbered
// pass-major: every item of pass p precedes every item of pass p + 1, so a CTA
// that takes an item of pass p + 1 can rely on all items of pass p having been
// taken by running CTAs, which never wait on later passes: the queue cannot
// deadlock. Before starting an item of pass p > 0 a CTA waits until all tiles
// of pass p - 1 of the same (instance, family) are complete (a counter per pair,
// incremented after a fence). The wait is bounded by a time limit after which
// the kernel records QLA_ETIMEOUT, stops taking items and returns.
//
// A lattice offers only its own tiles until its pass completes, so the tiles
// are low enough for the batch together to fill the GPU (batch_rows). Ten lattices
// of sides 256 to 1024, 400 steps: 110 ms with tiles of up to 768 rows of the
// shared-memory sweep (15 G site-updates/s, most SMs idle), 21 ms now (78 G).
#include <math.h>
#include <string.h>

#include <algorithm>
#include <numeric>
#include <string>
#include <vector>

#include "../../include/qla.h"
#include "qla_march.cuh"

namespace qla {

struct BatchInst {
    char *q[2];
    const char *rec[2];             // per family
    const unsigned char *flags[2];
    int Nx, Ny, w_valid, halo, strips, chunks;
    int tiles;                      // per pass and family
    int passes;                     // of kBatchSteps steps
    int wide;                       // its rotations take the form for any angle (MODE_WIDE)
};

// A lattice whose records are not worth their memory, or do not fit: coefficients in
// pair planes, advanced by the shared-memory sweep, whose passes follow the batch
// kernel in the graph. Its state returns to q[0] after every run.
struct BatchPlanes {
    void *q[2];
    const void *coef;
    int Nx, Ny, chunk, mode;
    int K;                          // steps per pass
    int ctas;                       // balanced split (chunk = 0)
    long long passes;
};

struct BatchSched {
    const BatchInst *inst;           // sorted by passes, descending
    int ninst;
    int maxpass;
    const long long *pass_start;     // [maxpass + 1]
    const int *active_count;         // [maxpass]: instances with passes > p (a prefix of inst)
    const long long *tile_prefix;    // [ninst + 1]: prefix sums of 2 * tiles
    unsigned long long *next;        // work counter
    unsigned int *done;              // [2 * ninst] completed tiles per (instance, family)
    int *cur;                        // [ninst] state buffer holding the input of pass 0
    int *error;                      // set to 1 on a wait timeout
    long long timeout_ns;
    unsigned int withhold;           // test hook: extra completions a dependency waits for (0 normally)
};

// The marching configuration of the batch: two steps per pass.
constexpr int kBatchSteps = 2;
constexpr int BC = 4, BD = 3, BU = 4, BWPC = 4, BMINB = 2;

// Largest k in [0, n) with a[k] <= v (a ascending, a[0] <= v): 32 candidates
// per round, one dependent load each, by a whole warp.
__device__ __forceinline__ int warp_search(const long long *a, int n, long long v, int lane) {
    int lo = 0;
    while (n > 1) {
        const int step = (n + 31) / 32;
        const int k = lane * step;
        const bool le = k < n && a[lo + k] <= v;
        const int last = 31 - __clz(int(__ballot_sync(0xffffffffu, le) | 1u));
        lo += last * step;
        n = min(step, n - last * step);
    }
    return lo;
}

// MODE with MODE_WIDE: some lattice of the batch (BatchInst::wide) rotates in that
// form, the others as without it.
template <bool INTER, int MODE, bool VEC>
__global__ void __launch_bounds__(32 * BWPC, BMINB) batch_kernel(const BatchSched S) {
    using L = MarchLayout<float, BC, kBatchSteps, BD, INTER>;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    __shared__ MarchArgs args;  // the item's lattice and family (entry 0)
    __shared__ int item[5];     // stop, instance, family, tile, wide
    const int lane = threadIdx.x & 31;
    const int warp = __shfl_sync(0xffffffffu, int(threadIdx.x) >> 5, 0);
    for (;;) {
        if (warp == 0) {
            unsigned long long g = 0;
            if (lane == 0) g = atomicAdd(S.next, 1ull);
            g = __shfl_sync(0xffffffffu, g, 0);
            int stop = g >= (unsigned long long)S.pass_start[S.maxpass] || *(volatile int *)S.error ? 1 : 0;
            int inst = 0, fam = 0, tile = 0, wide = 0;
            if (!stop) {
                const int pass = warp_search(S.pass_start, S.maxpass, (long long)g, lane);
                const long long r = (long long)g - S.pass_start[pass];
                inst = warp_search(S.tile_prefix, S.active_count[pass], r, lane);
                const BatchInst &I = S.inst[inst];
                const int rr = int(r - S.tile_prefix[inst]);
                const int tiles = I.tiles;
                if constexpr (MODE & MODE_WIDE) wide = I.wide;
                fam = rr / tiles;
                tile = rr % tiles;
                if (lane == 0) {
                    const int par = (S.cur[inst] + pass) & 1;
                    args.fam[0] = march_fam<float>(I.q[par], I.q[par ^ 1], I.rec[fam], I.flags[fam], fam, I.Nx, I.Ny);
                    args.Nx = I.Nx;
                    args.Ny = I.Ny;
                    args.w_valid = I.w_valid;
                    args.halo = I.halo;
                    args.strips = I.strips;
                    args.chunks = I.chunks;
                    if (pass > 0) {
                        const unsigned int target = (unsigned int)pass * (unsigned int)tiles + S.withhold;
                        const unsigned long long t0 = global_ns();
                        while (int(ld_acquire_u32(&S.done[2 * inst + fam]) - target) < 0) {
                            if (*(volatile int *)S.error) {  // another CTA gave up: stop as well
                                stop = 1;
                                break;
                            }
                            if ((long long)(global_ns() - t0) > S.timeout_ns) {
                                atomicExch(S.error, 1);
                                stop = 1;
                                break;
                            }
                            __nanosleep(64);
                        }
                    }
                }
                stop = __shfl_sync(0xffffffffu, stop, 0);
            }
            if (lane == 0) {
                item[0] = stop;
                item[1] = inst;
                item[2] = fam;
                item[3] = tile;
                item[4] = wide;
            }
        }
        __syncthreads();
        if (item[0]) break;
        const int w = item[3] * BWPC + warp;
        if (w < args.strips * args.chunks) {
            const int strip = w % args.strips, chunk = w / args.strips;
            const int y0 = int((long long)args.Ny * chunk / args.chunks);
            const int y1 = int((long long)args.Ny * (chunk + 1) / args.chunks);
            constexpr int NARROW = MODE & ~MODE_WIDE;
            if ((MODE & MODE_WIDE) && item[4])
                march_share<float, BC, kBatchSteps, BD, BU, INTER, MODE, VEC, false>(args, args.fam[0], strip, y0, y1,
                                                                                   smem_raw + warp * L::WARP, lane);
            else
                march_share<float, BC, kBatchSteps, BD, BU, INTER, NARROW, VEC, false>(args, args.fam[0], strip, y0, y1,
                                                                                     smem_raw + warp * L::WARP, lane);
        }
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0) {
            __threadfence();
            atomicAdd(&S.done[2 * item[1] + item[2]], 1u);
        }
        __syncthreads();  // the item's words are read before the next item overwrites them
    }
}

// After a run every instance has advanced `passes` passes: flip its parity.
__global__ void batch_flip(const BatchInst *inst, int *cur, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) cur[i] ^= (inst[i].passes & 1);
}

cudaError_t launch_planes(const BatchPlanes &p, bool inter, int *error, cudaStream_t st) {
    SweepArgs a{};
    a.coef = p.coef;
    a.Nx = p.Nx;
    a.Ny = p.Ny;
    a.w_valid = sweep_strip_width() - 8 * p.K;
    a.chunk = p.chunk;
    a.ctas = p.ctas;
    a.interleaved = inter ? 1 : 0;
    a.mode = p.mode;
    a.vec = 1;  // Nx is a multiple of 4
    a.error = error;
    for (long long i = 0; i < p.passes; ++i) {
        a.q_in = p.q[i & 1];
        a.q_out = p.q[(i + 1) & 1];
        const cudaError_t e = launch_sweep_f32(p.K, a, 2, st);
        if (e != cudaSuccess) return e;
    }
    return p.passes & 1 ? cudaMemcpyAsync(p.q[0], p.q[1], 24ull * p.Nx * p.Ny, cudaMemcpyDeviceToDevice, st)
                        : cudaSuccess;
}

// Sets the shared-memory attribute and returns the persistent grid size (SMs x
// resident CTAs); called before stream capture. With S: launches *grid CTAs.
template <bool INTER, int MODE, bool VEC>
cudaError_t batch_t(int sms, int *grid, const BatchSched *S, cudaStream_t st) {
    using L = MarchLayout<float, BC, kBatchSteps, BD, INTER>;
    constexpr int smem = L::WARP * BWPC;
    auto kern = batch_kernel<INTER, MODE, VEC>;
    if (S == nullptr) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
        int occ = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, 32 * BWPC, smem);
        if (e != cudaSuccess) return e;
        *grid = sms * (occ < 1 ? 1 : occ);
        return cudaSuccess;
    }
    kern<<<*grid, 32 * BWPC, smem, st>>>(*S);
    return cudaGetLastError();
}

// S == nullptr: prepare (attribute + grid size); otherwise launch with *grid CTAs.
// vec: every lattice's rows copy in vectors (march_vectors).
template <bool INTER, bool VEC>
cudaError_t batch_mode(int mode, int sms, int *grid, const BatchSched *S, cudaStream_t st) {
    switch (mode) {
        case 0: return batch_t<INTER, 0, VEC>(sms, grid, S, st);
        case MODE_UNITARY: return batch_t<INTER, MODE_UNITARY, VEC>(sms, grid, S, st);
        case MODE_UNITARY | MODE_WIDE: return batch_t<INTER, MODE_UNITARY | MODE_WIDE, VEC>(sms, grid, S, st);
    }
    return cudaErrorInvalidValue;
}
cudaError_t batch_dispatch(bool vec, bool inter, int mode, int sms, int *grid, const BatchSched *S, cudaStream_t st) {
    if (vec) return inter ? batch_mode<true, true>(mode, sms, grid, S, st) : batch_mode<false, true>(mode, sms, grid, S, st);
    return inter ? batch_mode<true, false>(mode, sms, grid, S, st) : batch_mode<false, false>(mode, sms, grid, S, st);
}

}  // namespace qla

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------

struct qla_batch {
    int n = 0;
    int K = 4;
    int dev = 0;
    int sms = 152;
    bool inter = true, vec = true;
    int mode = 0;  // SweepMode: MODE_WIDE if any lattice's
    cudaStream_t stream = nullptr;
    std::vector<qla::BatchInst> inst;  // sorted order
    std::vector<qla::BatchPlanes> planes;
    std::vector<int> order;            // order[k] = user index of sorted instance k
    std::vector<int> slot;             // slot[user index] = sorted position
    std::vector<int> cur;              // host copy of the parities
    std::vector<void *> allocs;
    qla::BatchInst *d_inst = nullptr;
    long long *d_pass_start = nullptr;
    int *d_active = nullptr;
    long long *d_tile_prefix = nullptr;
    unsigned long long *d_next = nullptr;
    unsigned int *d_done = nullptr;
    int *d_cur = nullptr;
    int *d_error = nullptr;
    void *d_scratch = nullptr;
    qla::DiagResult *d_diag = nullptr;
    qla::DiagResult *h_diag = nullptr;
    int maxpass = 0;
    int grid = 0;
    long long total_items = 0;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    long long timeout_ns = 4000000000LL;  // per dependency wait
    unsigned int withhold = 0;
    std::string msg;
};

namespace {

template <typename P>
cudaError_t dalloc(qla_batch *b, P **p, size_t bytes) {
    void *v = nullptr;
    cudaError_t e = cudaMalloc(&v, bytes);
    if (e == cudaSuccess) {
        b->allocs.push_back(v);
        *p = static_cast<P *>(v);
    }
    return e;
}

// Rows per share, at most: as many as let the batch's warps fill the GPU's slots (8
// per SM) a little more than once (a lattice's pass ends with its last tile; more,
// lower shares pay the march_delay(2) = 17 warm-up rows more often), and at least 8. Ten lattices of sides 256 to 1024,
// 400 steps: 16 rows 34.8 ms, 28 (filled twice) 23.9, 48 21.2, 64 22.2, 96 28.5;
// the three largest of them: 15 rows 16.5 ms, 32 14.1, 64 20.4.
int batch_rows(const std::vector<qla::MarchGeo> &geo, int sms) {
    double units = 0.0;
    for (const qla::MarchGeo &g : geo) units += 2.0 * g.strips * g.Ny;
    return std::max(8, int(units / (1.15 * 8.0 * sms) + 0.5));
}

}  // namespace

extern "C" {

qla_status qla_batch_create(int count, const qla_instance_desc *descs, const qla_options *opt, qla_batch **out) {
    if (!out || count < 1 || !descs) return QLA_EINVAL;
    *out = nullptr;
    qla_options o;
    qla_default_options(&o);
    if (opt) o = *opt;
    if (o.precision != QLA_FP32 || o.families != QLA_FAMILIES_BOTH) return QLA_EUNSUPPORTED;
    const int K = o.steps_per_pass > 0 ? o.steps_per_pass : 4;
    if (K != 2 && K != 4) return QLA_EUNSUPPORTED;
    std::vector<int> modes(count);
    std::vector<char> planes(count);  // on pair planes (BatchPlanes)
    std::vector<qla::MarchGeo> geo_of(count);
    size_t bytes = 0, index_bytes = 0;
    for (int i = 0; i < count; ++i) {
        const qla_instance_desc &d = descs[i];
        if (d.Nx < 4 || d.Ny < 1 || d.Nx % 4 != 0 || (long long)d.Nx * d.Ny > 2147483647LL) return QLA_EINVAL;
        if (!d.n_x || !d.n_y || !d.n_z || !(d.delta > 0.0) || !(d.delta <= 0.5)) return QLA_EINVAL;
        if (d.nsteps < 0 || d.nsteps % K != 0) return QLA_EINVAL;
        const size_t P = size_t(d.Nx) * d.Ny;
        const double *nn[3] = {d.n_x, d.n_y, d.n_z};
        bool ordinary = true;
        for (int k = 0; k < 3; ++k)
            if (!qla::index_valid(nn[k], P, &ordinary)) return QLA_EINVAL;
        modes[i] = qla::rotation_mode(nn, ordinary, d.Nx, d.Ny, d.delta, 0, o.sequence == QLA_SEQ_INTERLEAVED ? 1 : 0,
                                      o.potential == QLA_POT_UNITARY ? 1 : 0);
        const size_t pairs = size_t(qla::NCOEF) * P * 4;
        planes[i] = !qla::march_geometry(0, d.Nx, d.Ny, &geo_of[i]) || !qla::march_worth(geo_of[i], pairs);
        bytes += 48 * P + (planes[i] ? pairs : qla::march_bytes(geo_of[i], 2));
        index_bytes = std::max(index_bytes, 24 * P);
    }
    if (bytes + index_bytes > qla::kDeviceBytes) planes.assign(count, 1);
    qla_batch *b = new qla_batch();
    auto bail = [&](qla_status s) {
        qla_batch_destroy(b);
        return s;
    };
    b->n = count;
    b->K = K;
    b->inter = o.sequence == QLA_SEQ_INTERLEAVED;
    for (const int m : modes) b->mode |= m;
    if (o.device >= 0) {
        if (cudaSetDevice(o.device) != cudaSuccess) return bail(QLA_ECUDA);
        b->dev = o.device;
    } else if (cudaGetDevice(&b->dev) != cudaSuccess) {
        return bail(QLA_ECUDA);
    }
    cudaDeviceGetAttribute(&b->sms, cudaDevAttrMultiProcessorCount, b->dev);
    if (cudaStreamCreateWithFlags(&b->stream, cudaStreamNonBlocking) != cudaSuccess) return bail(QLA_ECUDA);

    // sort by number of passes, descending (active instances of a pass are a prefix;
    // lattices on pair planes take no part: the last)
    auto steps = [&](int i) { return planes[i] ? 0LL : descs[i].nsteps; };
    b->order.resize(count);
    std::iota(b->order.begin(), b->order.end(), 0);
    std::stable_sort(b->order.begin(), b->order.end(),
                     [&](int a, int c) { return steps(a) > steps(c); });
    b->slot.resize(count);
    for (int k = 0; k < count; ++k) b->slot[b->order[k]] = k;
    b->inst.resize(count);
    b->cur.assign(count, 0);
    size_t scratch_max = 0;
    std::vector<qla::MarchGeo> marching;
    for (int i = 0; i < count; ++i) {
        if (planes[i]) continue;
        marching.push_back(geo_of[i]);
        b->vec = b->vec && qla::march_vectors(geo_of[i]);
    }
    const int rows = batch_rows(marching, b->sms);
    for (int k = 0; k < count; ++k) {
        const qla_instance_desc &d = descs[b->order[k]];
        qla::BatchInst &I = b->inst[k];
        const qla::MarchGeo &g = geo_of[b->order[k]];
        const bool planar = planes[b->order[k]] != 0;
        const int mode = modes[b->order[k]];
        const size_t P = size_t(d.Nx) * d.Ny;
        I.Nx = d.Nx;
        I.Ny = d.Ny;
        I.w_valid = g.w_valid;
        I.halo = g.halo;
        I.strips = g.strips;
        // (a lattice's chunk_rows: at most, see march_plan; ten lattices of sides 256 to
        // 1024, 100 steps, 768 rows: 30 ms in tiles of the shared-memory sweep, 32 with
        // as many rows per warp, 5.8 now)
        const int ch = std::min(d.chunk_rows > 0 ? std::min(d.chunk_rows, rows) : rows, d.Ny);
        I.chunks = (d.Ny + ch - 1) / ch;
        I.tiles = (I.strips * I.chunks + qla::BWPC - 1) / qla::BWPC;
        I.passes = int(d.nsteps / qla::kBatchSteps);
        I.wide = mode & qla::MODE_WIDE ? 1 : 0;
        if (planar) I.passes = I.tiles = 0;
        float *q0, *q1;
        char *mem;
        double *idx;
        if (dalloc(b, &q0, 6 * P * 4) != cudaSuccess || dalloc(b, &q1, 6 * P * 4) != cudaSuccess ||
            dalloc(b, &mem, planar ? size_t(qla::NCOEF) * P * 4 : qla::march_bytes(g, 2)) != cudaSuccess ||
            dalloc(b, &idx, 3 * P * 8) != cudaSuccess) {
            cudaGetLastError();
            return bail(QLA_ENOMEM);
        }
        I.q[0] = reinterpret_cast<char *>(q0);
        I.q[1] = reinterpret_cast<char *>(q1);
        for (int f = 0; f < 2; ++f) {
            if (planar) {
                I.rec[f] = nullptr;
                I.flags[f] = nullptr;
                continue;
            }
            I.rec[f] = mem + f * g.record_bytes;
            I.flags[f] = reinterpret_cast<const unsigned char *>(mem + 2 * g.record_bytes + f * g.flag_bytes);
        }
        const double *nn[3] = {d.n_x, d.n_y, d.n_z};
        for (int c = 0; c < 3; ++c)
            if (cudaMemcpyAsync(idx + c * P, nn[c], P * 8, cudaMemcpyHostToDevice, b->stream) != cudaSuccess)
                return bail(QLA_ECUDA);
        const int inter = b->inter ? 1 : 0;
        if ((planar ? qla::launch_coefficients(idx, mem, d.Nx, d.Ny, d.delta, 0, inter, mode, b->stream)
                    : qla::launch_march_records(g, idx, mem, 2, 0, d.delta, 0, inter, mode, b->stream)) != cudaSuccess)
            return bail(QLA_ECUDA);
        if (planar) {
            qla::BatchPlanes p;
            p.q[0] = q0;
            p.q[1] = q1;
            p.coef = mem;
            p.Nx = d.Nx;
            p.Ny = d.Ny;
            p.chunk = d.chunk_rows > 0 ? std::min(d.chunk_rows, d.Ny) : 0;
            p.mode = mode;
            p.K = mode & qla::MODE_WIDE ? 1 : 2;
            const qla::SweepSplit sp = qla::make_sweep_split(d.Nx, d.Ny, p.K, qla::sweep_block_rows(0, p.K), 1);
            p.ctas = int(std::min((long long)b->sms * qla::sweep_occupancy_f32(p.K, inter), (long long)sp.nsx * d.Ny));
            p.passes = d.nsteps / p.K;
            b->planes.push_back(p);
        }
        if (cudaMemsetAsync(q0, 0, 6 * P * 4, b->stream) != cudaSuccess ||
            cudaMemsetAsync(q1, 0, 6 * P * 4, b->stream) != cudaSuccess)
            return bail(QLA_ECUDA);
        if (d.pulse_polarization == QLA_POL_EZ || d.pulse_polarization == QLA_POL_EY) {
            if (!(d.pulse_sigma > 0.0)) return bail(QLA_EINVAL);
            if (qla::launch_init_pulse(q0, d.Nx, d.Ny, 0, d.pulse_polarization, d.pulse_x0, d.pulse_sigma,
                                       d.pulse_amplitude, b->stream) != cudaSuccess)
                return bail(QLA_ECUDA);
        }
        scratch_max = std::max(scratch_max, qla::diag_scratch_bytes(d.Nx, d.Ny));
        // the index fields are only needed for the coefficients
        if (cudaStreamSynchronize(b->stream) != cudaSuccess) return bail(QLA_ECUDA);
        cudaFree(idx);
        b->allocs.pop_back();
    }
    // schedule tables
    b->maxpass = b->inst[0].passes;
    std::vector<long long> tile_prefix(count + 1, 0);
    for (int k = 0; k < count; ++k) tile_prefix[k + 1] = tile_prefix[k] + 2LL * b->inst[k].tiles;
    std::vector<long long> pass_start(b->maxpass + 1, 0);
    std::vector<int> active(std::max(1, b->maxpass), 0);
    for (int p = 0; p < b->maxpass; ++p) {
        int a = 0;
        while (a < count && b->inst[a].passes > p) ++a;
        active[p] = a;
        pass_start[p + 1] = pass_start[p] + tile_prefix[a];
    }
    b->total_items = pass_start[b->maxpass];
    if (dalloc(b, &b->d_inst, sizeof(qla::BatchInst) * count) != cudaSuccess ||
        dalloc(b, &b->d_pass_start, sizeof(long long) * (b->maxpass + 1)) != cudaSuccess ||
        dalloc(b, &b->d_active, sizeof(int) * active.size()) != cudaSuccess ||
        dalloc(b, &b->d_tile_prefix, sizeof(long long) * (count + 1)) != cudaSuccess ||
        dalloc(b, &b->d_next, 64) != cudaSuccess || dalloc(b, &b->d_done, sizeof(unsigned) * 2 * count) != cudaSuccess ||
        dalloc(b, &b->d_cur, sizeof(int) * count) != cudaSuccess || dalloc(b, &b->d_error, 64) != cudaSuccess ||
        dalloc(b, &b->d_scratch, scratch_max + 512) != cudaSuccess)
        return bail(QLA_ENOMEM);
    b->d_diag = reinterpret_cast<qla::DiagResult *>(static_cast<char *>(b->d_scratch) + ((scratch_max + 255) / 256) * 256);
    if (cudaMallocHost(reinterpret_cast<void **>(&b->h_diag), sizeof(qla::DiagResult)) != cudaSuccess)
        return bail(QLA_ENOMEM);
    if (cudaMemcpy(b->d_inst, b->inst.data(), sizeof(qla::BatchInst) * count, cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(b->d_pass_start, pass_start.data(), sizeof(long long) * pass_start.size(), cudaMemcpyHostToDevice) !=
            cudaSuccess ||
        cudaMemcpy(b->d_active, active.data(), sizeof(int) * active.size(), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(b->d_tile_prefix, tile_prefix.data(), sizeof(long long) * tile_prefix.size(),
                   cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemset(b->d_cur, 0, sizeof(int) * count) != cudaSuccess)
        return bail(QLA_ECUDA);
    if (qla::batch_dispatch(b->vec, b->inter, b->mode, b->sms, &b->grid, nullptr, nullptr) != cudaSuccess)
        return bail(QLA_ECUDA);
    *out = b;
    return QLA_OK;
}

qla_status qla_batch_run(qla_batch *b) {
    if (!b) return QLA_EINVAL;
    if (cudaSetDevice(b->dev) != cudaSuccess) return QLA_ECUDA;
    if (!b->exec) {
        qla::BatchSched S;
        S.inst = b->d_inst;
        S.ninst = b->n;
        S.maxpass = b->maxpass;
        S.pass_start = b->d_pass_start;
        S.active_count = b->d_active;
        S.tile_prefix = b->d_tile_prefix;
        S.next = b->d_next;
        S.done = b->d_done;
        S.cur = b->d_cur;
        S.error = b->d_error;
        S.timeout_ns = b->timeout_ns;
        S.withhold = b->withhold;
        if (cudaStreamBeginCapture(b->stream, cudaStreamCaptureModeThreadLocal) != cudaSuccess) return QLA_ECUDA;
        cudaError_t e = cudaMemsetAsync(b->d_next, 0, 64, b->stream);
        if (e == cudaSuccess) e = cudaMemsetAsync(b->d_done, 0, sizeof(unsigned) * 2 * b->n, b->stream);
        if (e == cudaSuccess) e = cudaMemsetAsync(b->d_error, 0, 64, b->stream);
        if (e == cudaSuccess && b->maxpass > 0)
            e = qla::batch_dispatch(b->vec, b->inter, b->mode, b->sms, &b->grid, &S, b->stream);
        for (const qla::BatchPlanes &p : b->planes)
            if (e == cudaSuccess) e = qla::launch_planes(p, b->inter, b->d_error, b->stream);
        if (e == cudaSuccess) {
            qla::batch_flip<<<(b->n + 127) / 128, 128, 0, b->stream>>>(b->d_inst, b->d_cur, b->n);
            e = cudaGetLastError();
        }
        cudaGraph_t g = nullptr;
        const cudaError_t e2 = cudaStreamEndCapture(b->stream, &g);
        if (e != cudaSuccess || e2 != cudaSuccess) {
            if (g) cudaGraphDestroy(g);
            b->msg = std::string("graph capture failed: ") + cudaGetErrorString(e != cudaSuccess ? e : e2);
            return QLA_ECUDA;
        }
        b->graph = g;
        if (cudaGraphInstantiate(&b->exec, g, 0) != cudaSuccess) {
            b->msg = "graph instantiation failed";
            return QLA_ECUDA;
        }
    }
    if (cudaGraphLaunch(b->exec, b->stream) != cudaSuccess) return QLA_ECUDA;
    int err = 0;
    if (cudaMemcpyAsync(&err, b->d_error, sizeof(int), cudaMemcpyDeviceToHost, b->stream) != cudaSuccess ||
        cudaStreamSynchronize(b->stream) != cudaSuccess)
        return QLA_ECUDA;
    for (int k = 0; k < b->n; ++k) b->cur[k] ^= (b->inst[k].passes & 1);
    if (err) {
        b->msg = "a dependency wait or a wait for row copies timed out";
        return QLA_ETIMEOUT;
    }
    return QLA_OK;
}

qla_status qla_batch_get_fields_f32(qla_batch *b, int i, float *q) {
    if (!b || i < 0 || i >= b->n || !q) return QLA_EINVAL;
    if (cudaSetDevice(b->dev) != cudaSuccess) return QLA_ECUDA;
    const int k = b->slot[i];
    const qla::BatchInst &I = b->inst[k];
    const size_t P = size_t(I.Nx) * I.Ny;
    if (cudaMemcpyAsync(q, I.q[b->cur[k]], 6 * P * 4, cudaMemcpyDeviceToHost, b->stream) != cudaSuccess ||
        cudaStreamSynchronize(b->stream) != cudaSuccess)
        return QLA_ECUDA;
    return QLA_OK;
}

qla_status qla_batch_diagnostics(qla_batch *b, int i, qla_diag *out) {
    if (!b || i < 0 || i >= b->n || !out) return QLA_EINVAL;
    if (cudaSetDevice(b->dev) != cudaSuccess) return QLA_ECUDA;
    const int k = b->slot[i];
    const qla::BatchInst &I = b->inst[k];
    if (qla::launch_diagnostics(I.q[b->cur[k]], 0, I.Nx, I.Ny, b->d_scratch, b->d_diag, b->stream) != cudaSuccess ||
        cudaMemcpyAsync(b->h_diag, b->d_diag, sizeof(qla::DiagResult), cudaMemcpyDeviceToHost, b->stream) !=
            cudaSuccess ||
        cudaStreamSynchronize(b->stream) != cudaSuccess)
        return QLA_ECUDA;
    out->energy = b->h_diag->energy_sum / (double(I.Nx) * I.Ny);
    out->div_l2_sq = b->h_diag->div_sq_sum;
    out->div_max = b->h_diag->div_max;
    out->b_max = b->h_diag->b_max;
    out->nonfinite = (long long)b->h_diag->nonfinite;
    return out->nonfinite ? QLA_ENONFINITE : QLA_OK;
}

qla_status qla_batch_info(const qla_batch *b, long long *total_items, int *steps_per_pass, long long *site_updates) {
    if (!b) return QLA_EINVAL;
    if (total_items) *total_items = b->total_items;
    if (steps_per_pass) *steps_per_pass = b->K;
    if (site_updates) {
        long long s = 0;
        for (const auto &I : b->inst) s += (long long)I.Nx * I.Ny * I.passes * qla::kBatchSteps;
        for (const auto &p : b->planes) s += (long long)p.Nx * p.Ny * p.passes * p.K;
        *site_updates = s;
    }
    return QLA_OK;
}

qla_status qla_batch_set_wait_limit(qla_batch *b, long long timeout_ns, int withhold) {
    if (!b || timeout_ns <= 0 || withhold < 0) return QLA_EINVAL;
    b->timeout_ns = timeout_ns;
    b->withhold = (unsigned int)withhold;
    if (b->exec) cudaGraphExecDestroy(b->exec);
    if (b->graph) cudaGraphDestroy(b->graph);
    b->exec = nullptr;
    b->graph = nullptr;
    return QLA_OK;
}

const char *qla_batch_last_error(const qla_batch *b) { return b ? b->msg.c_str() : "NULL batch"; }

void qla_batch_destroy(qla_batch *b) {
    if (!b) return;
    cudaSetDevice(b->dev);
    if (b->stream) cudaStreamSynchronize(b->stream);
    if (b->exec) cudaGraphExecDestroy(b->exec);
    if (b->graph) cudaGraphDestroy(b->graph);
    for (void *p : b->allocs) cudaFree(p);
    if (b->h_diag) cudaFreeHost(b->h_diag);
    if (b->stream) cudaStreamDestroy(b->stream);
    cudaGetLastError();
    delete b;
}

}  // extern "C"
