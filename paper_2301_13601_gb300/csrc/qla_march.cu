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
    // 32-bit byte offsets in a plane; strips * Ny shares at most
    return (unsigned long long)Nx * Ny * g->es < (1ull << 32) && (long long)g->strips * Ny < (1LL << 30);
}

size_t march_bytes(const MarchGeo &g, int nfam) { return size_t(nfam) * (g.record_bytes + g.flag_bytes); }

namespace {

// Row ranges per strip. One warp each, `slots` resident at a time over the
// families together. A single wave ends with its slowest warp (the rows whose
// V angles are nonzero cost more, measured up to a quarter over the mean);
// several waves even that out at the price of march_delay(K) more rows per
// share. FP32, two steps, GB300 (us per step): 8192^2 8 row ranges (one wave)
// 739, 16 678, 32 628, 64 639; 4096^2 16 (one wave) 160, 32 155, 64 165.
int march_chunks(const MarchGeo &g, int nfam, int delay, int slots) {
    const double strips = double(g.strips) * nfam;
    int best = 1;
    double cost = 1e300;
    for (int n = 1; n <= g.Ny; ++n) {
        const double share = double((g.Ny + n - 1) / n + delay);
        const double waves = strips * n / slots;
        const double c = waves <= 1.0 ? 1.25 * share : waves * share + 0.6 * share;
        if (c < cost) {
            cost = c;
            best = n;
        }
        if (waves > 32.0) break;
    }
    return best;
}

}  // namespace

void march_plan(MarchGeo *g, int nfam, int chunk, int sms) {
    for (int K = 1; K <= 2; ++K)
        g->chunks[K] = chunk > 0 ? (g->Ny + chunk - 1) / chunk
                                 : march_chunks(*g, nfam, march_delay(K), sms * (K == 2 ? 8 : 12));
    g->chunks[0] = 0;
}

cudaError_t launch_march(const MarchGeo &g, int K, const void *q_in, void *q_out, const void *mem, int nfam, int fam0,
                         int interleaved, int unitary, cudaStream_t st) {
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
    a.chunks = g.chunks[K];
    // the lane's columns as one vector: 4 (FP32) or 2 (FP64) columns
    const bool vec = g.Nx % (f64 ? 2 : 4) == 0;
    if (f64) return vec ? launch_march_f64_k1(a, nfam, interleaved, unitary, st)
                        : launch_march_f64_k1_any(a, nfam, interleaved, unitary, st);
    if (K == 2) return vec ? launch_march_f32_k2(a, nfam, interleaved, unitary, st)
                           : launch_march_f32_k2_any(a, nfam, interleaved, unitary, st);
    return vec ? launch_march_f32_k1(a, nfam, interleaved, unitary, st)
               : launch_march_f32_k1_any(a, nfam, interleaved, unitary, st);
}

}  // namespace qla
