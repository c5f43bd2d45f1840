// Steps, fields and diagnostics of a lattice (FP32 storage here, 16-bit in
// cmrt_step16.cu), and the rows per CTA of the march.
#include "cmrt_march.cuh"

namespace cmrt {
namespace {

__global__ void k_diag_reduce(const double* __restrict__ partials, int nblocks, double* __restrict__ out) {
    pdl_begin();
    __shared__ double red[kThreads / 32][kDiagSlots];
    double v[kDiagSlots] = {0, 0, 0, 0, 0, 0};
    for (int b = threadIdx.x; b < nblocks; b += blockDim.x) {
#pragma unroll
        for (int j = 0; j < kDiagSlots; ++j) {
            const double o = partials[static_cast<size_t>(b) * kDiagSlots + j];
            v[j] = (j == 4) ? fmax(v[j], o) : v[j] + o;
        }
    }
#pragma unroll
    for (int j = 0; j < kDiagSlots; ++j) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            const double o = __shfl_down_sync(0xffffffffu, v[j], off);
            v[j] = (j == 4) ? fmax(v[j], o) : v[j] + o;
        }
    }
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0) {
#pragma unroll
        for (int j = 0; j < kDiagSlots; ++j) red[warp][j] = v[j];
    }
    __syncthreads();
    if (threadIdx.x < kDiagSlots) {
        double acc = red[0][threadIdx.x];
        for (int w = 1; w < kThreads / 32; ++w) {
            const double o = red[w][threadIdx.x];
            acc = (threadIdx.x == 4) ? fmax(acc, o) : acc + o;
        }
        out[threadIdx.x] = acc;
    }
}

}  // namespace

size_t state_node_bytes(int precision) {
    return precision == kPrecF32 ? kPlanes * 4 : Layout16<__half2>::node_bytes();
}

dim3 chain_grid(int nx, int ny, int rows) {
    return dim3(static_cast<unsigned>((nx + kTileX - 1) / kTileX), static_cast<unsigned>((ny + rows - 1) / rows), 1);
}

int chain_rows(int nx, int ny, int sms, int precision) {
    // Rows per CTA.  A CTA spends rows + 7 row iterations (7 fill the pipeline; with
    // 16-bit storage ten, of which three only decode and count as two: with a fill of
    // ten FP16 4096 x 2048 takes 271 us instead of 265, 774 x 2786 113 instead of 105,
    // 1308 x 623 36 instead of 33; 6902 x 648 196 instead of 201, BF16 4488 x 6270 847
    // instead of 868); an iteration takes longer the more CTAs share its SM: 0.79,
    // 0.95, 1.40 and 1.47 us with one to four (FP32, states within L2; 16-bit storage
    // goes by the same ratios).  Within one wave the fullest SM sets the time, by a
    // quarter more where the state is beyond L2 (2048^2: 120 us with 64 rows in one
    // wave, 129 with 32; 4096^2: 505 us with 241 rows, 435 with 64).  Past one wave the
    // hardware hands out CTAs as others finish, which evens out the SMs'
    // different speeds (two dies), and half a CTA's time is lost at the end.
    // Measured at 8192^2: 36.3, 38.0, 40.4, 40.6, 40.9, 40.5 and 39.5 GLUPS with
    // 512, 256, 192, 128, 96, 64 and 48 rows; at 4096^2 26.8, 32.8, 36.1, 37.8,
    // 38.2, 38.2 and 37.3 with 512, 256, 128, 96, 64, 48 and 32.
    constexpr double kUs[4] = {0.79, 0.95, 1.40, 1.47};
    static_assert(march_ctas<kWin>() == 4, "a time per CTA count");
    const int strips = (nx + kTileX - 1) / kTileX;
    const int n_sms = sms > 0 ? sms : 1;
    const int fill = precision == kPrecF32 ? 7 : 9;
    const double slots = 4.0 * n_sms;
    const bool beyond_l2 = 144.0 * nx * ny > 126e6;
    int best = 8;
    double best_cost = -1.0;
    for (int rows = 1; rows <= 512; rows += rows < 32 ? 1 : 8) {
        const long ctas = static_cast<long>(strips) * ((ny + rows - 1) / rows);
        const double waves = ctas / slots;
        const double cost = (rows + fill) * (waves <= 1.0 ? kUs[(ctas - 1) / n_sms] * (beyond_l2 ? 1.25 : 1.0)
                                                          : kUs[3] * (waves + 0.5));
        if (best_cost < 0.0 || cost < best_cost) {
            best_cost = cost;
            best = rows;
        }
        if (rows >= ny) break;
    }
    return best;
}

cudaError_t launch_step(const void* src, void* dst, const StepParams& P, int rows, unsigned* flag, cudaStream_t s) {
    if (P.precision != kPrecF32) return launch_step16(src, dst, P, rows, flag, s);
    return launch_march<MarchF32<kWin>, Pass::Step>(src, dst, P, rows, FieldOut{}, flag, nullptr, s);
}

cudaError_t launch_step_fields(const float* src, float* dst, const StepParams& P, int rows, unsigned* flag,
                               float* fwd, cudaStream_t s) {
    FieldOut fo{};
    fo.fwd = fwd;
    return launch_march<MarchF32<kWin>, Pass::StepFields>(src, dst, P, rows, fo, flag, nullptr, s);
}

cudaError_t launch_fwd_fields(const float* src, const StepParams& P, float* fwd, cudaStream_t s) {
    FieldOut fo{};
    fo.fwd = fwd;
    return launch_small_any<MarchF32<kWin>, Pass::FwdFields>(src, nullptr, P, fo, nullptr, s);
}

cudaError_t launch_fields(const void* src, const StepParams& P, int rows, FieldOut out, bool host, cudaStream_t s) {
    // Page-locked outputs of an odd width: strips share 32-byte sectors, which fewer, longer
    // segments write closer together in time.  4095 x 1024 651 -> 609 us (581 before the
    // march), 701^2 87 -> 82 (80), FP16 4095 x 1024 660 -> 596 (593); not small lattices
    // (FP16 701^2 85 -> 94)
    if (host && P.nx % 4 != 0 && static_cast<long>(P.nx) * P.ny > (P.precision == kPrecF32 ? 400000 : 600000)) rows *= 4;
    if (P.precision != kPrecF32) return launch_fields16(src, P, rows, out, s);
    // 4-byte copies (nx no multiple of 4) in one wave of long segments: half the rows, in
    // two waves, even out the SMs.  4095 x 1024 148 -> 128 us, 3001 x 2000 204 -> 173;
    // not segments of 32 rows (1501 x 1500 77 -> 80) or several waves (6001 x 3001 473 -> 499)
    const dim3 g = chain_grid(P.nx, P.ny, rows);
    if (!host && P.nx % 4 != 0 && rows > 48 && static_cast<long>(g.x) * g.y <= 4 * 152) rows /= 2;
    return launch_march<MarchF32<kWin>, Pass::Fields>(src, nullptr, P, rows, out, nullptr, nullptr, s);
}

cudaError_t launch_diag_partials(const void* src, const StepParams& P, int rows, double* partials, cudaStream_t s) {
    if (P.precision != kPrecF32) return launch_diag_partials16(src, P, rows, partials, s);
    return launch_march<MarchF32<kWin>, Pass::Diag>(src, nullptr, P, rows, FieldOut{}, nullptr, partials, s);
}

cudaError_t launch_diag_partials_pre(const float* pre, const StepParams& P, int rows, double* partials,
                                     cudaStream_t s) {
    return launch_march<MarchF32<kWin>, Pass::Diag, true>(pre, nullptr, P, rows, FieldOut{}, nullptr, partials, s);
}

cudaError_t launch_diag_reduce(const double* partials, int nblocks, double* out, cudaStream_t s) {
    return launch_pdl(k_diag_reduce, dim3(1), dim3(kThreads), 0, s, partials, nblocks, out);
}

}  // namespace cmrt
