// Marching form of the sweep: geometry, share heights and dispatch (the kernels
// are in qla_march.cuh, the records in qla_coeffs.cu).
#include <algorithm>

#include "qla_march.cuh"

namespace qla {

bool march_geometry(int precision, int Nx, int Ny, MarchGeo *g) {
    g->Nx = Nx;
    g->Ny = Ny;
    g->es = precision ? 8 : 4;
    g->W = precision ? 64 : 128;
    g->halo = precision ? 4 : 8;
    g->w_valid = g->W - 2 * g->halo;
    g->strips = (Nx + g->w_valid - 1) / g->w_valid;
    g->record_bytes = size_t(g->strips) * (size_t(MARCH_ABOVE) + Ny + MARCH_BELOW) * MARCH_FIELDS * g->W * g->es;
    g->flag_bytes = (size_t(g->strips) * Ny + 255) / 256 * 256;
    return (long long)g->strips * Ny < (1LL << 30);  // shares, at most
}

bool march_worth(const MarchGeo &g, size_t pairs) {
    return march_bytes(g, 2) <= std::max(size_t(1) << 30, 4 * pairs);
}

bool march_vectors(const MarchGeo &g) {
    return g.Nx % (16 / g.es) == 0 && (unsigned long long)g.Nx * g.Ny * g.es < (1ull << 32);
}

size_t march_bytes(const MarchGeo &g, int nfam) { return size_t(nfam) * (g.record_bytes + g.flag_bytes); }

namespace {

// Row ranges per strip (one warp each). An iteration of a warp takes `lat`
// alone on its scheduler and `busy` of the scheduler's time (us, measured on
// GB300: FP32 from runs at 256^2 to 8192^2, FP64 from its pipe, which takes a
// warp instruction in 64 cycles). A pass alone on the GPU lasts as long as its
// most loaded SM; with others it costs the scheduler time it uses. Few ranges
// leave schedulers idle, many pay the march_delay(K) iterations before a
// range's first output row once more each: the sum of the two is minimised.
// CTAs of four warps load an SM's four schedulers evenly. A pass of one wave
// ends with its slowest warp (rows with nonzero V angles cost more): 1.35 times
// the mean at worst; more waves even out. us per step, three contexts in turn /
// one alone: 256^2 rows 1, 4, 16: 7.1/12.3, 4.1/10.3, 6.0/16.4; 2048^2 rows 32,
// 64, 128: 49.7/59.9, 39.8/52.0, 36.3/64.6; 8192^2 rows 128, 256, 1024:
// 532/565, 501/552, 483/620; FP64 256^2 rows 2, 8, 16: 150/221, 78/129, 64/192.
struct MarchCost {
    int resident;  // CTAs per SM
    double lat, busy;
};
constexpr MarchCost kMarchCost[3] = {{3, 5.2, 5.2}, {3, 0.55, 0.32}, {2, 0.89, 0.62}};  // FP64, FP32 K = 1, K = 2
constexpr double kLaunchUs = 3.0;

int march_chunks(const MarchGeo &g, int nfam, int K, int sms) {
    const MarchCost m = kMarchCost[g.es == 8 ? 0 : K];
    int best = 1;
    double cost = 1e300;
    for (int n = 1; n <= g.Ny; ++n) {
        const double its = double((g.Ny + n - 1) / n + march_delay(K));
        const long long ctas = (long long)nfam * (((long long)g.strips * n + 3) / 4);
        const long long per_sm = (ctas + sms - 1) / sms;
        const double busy = double(g.strips) * nfam * n * its * m.busy / (4.0 * sms);
        const double alone = per_sm <= m.resident
                                 ? 1.35 * its * (m.lat > per_sm * m.busy ? m.lat : per_sm * m.busy)
                                 : busy + 0.6 * its * m.resident * m.busy;
        const double c = kLaunchUs + alone + busy;
        if (c < cost) {
            cost = c;
            best = n;
        }
        if (per_sm > 32LL * m.resident) break;
    }
    return best;
}

}  // namespace

void march_plan(MarchGeo *g, int nfam, int chunk, int sms) {
    for (int K = 1; K <= 2; ++K) {
        g->chunks[K] = march_chunks(*g, nfam, K, sms);
        // A caller's rows are those of a tile, which a CTA of the shared-memory sweep
        // took (and whose best heights were 64 to 1024): a warp alone that swept as
        // many would leave the GPU to few warps (us per step, shared-memory sweep /
        // that many rows per warp / this: 256^2 256 rows 101 / 134 / 9, 1024^2 256
        // rows 97 / 111 / 24, 4096^2 1024 rows 343 / 380 / 157).
        if (chunk > 0) g->chunks[K] = std::max(g->chunks[K], (g->Ny + chunk - 1) / chunk);
    }
    g->chunks[0] = 0;
}

cudaError_t launch_march(const MarchGeo &g, int K, const void *q_in, void *q_out, const void *mem, int nfam, int fam0,
                         int interleaved, int mode, bool chained, cudaStream_t st) {
    const bool f64 = g.es == 8;
    if (!(K == 1 || (K == 2 && !f64))) return cudaErrorInvalidValue;
    MarchArgs a;
    const char *m = static_cast<const char *>(mem);
    for (int z = 0; z < 2; ++z) {
        const int k = std::min(z, nfam - 1);
        const void *rec = m + k * g.record_bytes;
        const unsigned char *flags = reinterpret_cast<const unsigned char *>(m + nfam * g.record_bytes + k * g.flag_bytes);
        a.fam[z] = f64 ? march_fam<double>(q_in, q_out, rec, flags, fam0 + k, g.Nx, g.Ny)
                       : march_fam<float>(q_in, q_out, rec, flags, fam0 + k, g.Nx, g.Ny);
    }
    a.Nx = g.Nx;
    a.Ny = g.Ny;
    a.w_valid = g.w_valid;
    a.halo = g.halo;
    a.strips = g.strips;
    a.ctas_fam = 0;
    a.chained = chained ? 1 : 0;
    a.chunks = g.chunks[K];
    const bool vec = march_vectors(g);
    if (f64) return vec ? launch_march_f64_k1(a, nfam, interleaved, mode, st)
                        : launch_march_f64_k1_any(a, nfam, interleaved, mode, st);
    if (K == 2) return vec ? launch_march_f32_k2(a, nfam, interleaved, mode, st)
                           : launch_march_f32_k2_any(a, nfam, interleaved, mode, st);
    return vec ? launch_march_f32_k1(a, nfam, interleaved, mode, st)
               : launch_march_f32_k1_any(a, nfam, interleaved, mode, st);
}

}  // namespace qla
