// The step, fields and diagnostics with App. B's order-6 colour and Phi'
// gradients (arXiv 2005.04642), FP32 storage:
//   d_a X = sum_N a_N sum_i w_i X(r + N c_i) c_ia,  (a_1, a_2, a_3) = (9/2, -9/10, 1/10),
// a stencil of radius 3, with the compact one for K and div u.
//
// One node per thread: a CTA takes a window of 32 x H nodes, 22 x (H - 10) of
// them its own (all H rows of a lattice of at most 32), gathers each node's populations into registers and runs
//   moments, chi, Phi' | grad rho^N (halo 2) | K, G, u (halo 1) | the rest,
// with a barrier between, the fields that a stencil reads in shared memory.
// What bounds it: the launch and one load latency on small lattices, else
// latency at one CTA of 1024 threads per SM (the window's halo makes the moments
// 2x, H = 32, to 4x their work; whole warps of halo rows skip the collision).
// Per step, as four passes over planes in memory -> here: 64^2 9.2 -> 2.8 us,
// 256^2 11.2 -> 5.4, 512^2 21.4 -> 19.3, 1024 x 512 38.2 -> 36.4, 2048^2 302 ->
// 296; one launch instead of four, and no 28 planes of scratch per node.  The same
// bits as the passes: a node's K takes the n-hat of its neighbours from their
// gradients (n-hat kept in shared memory instead: 1024 x 512 34.2 us, but the
// contraction of K then differs, and with walls the small u_y by 2e-4).
#include <atomic>

#include "cmrt_device.cuh"

namespace cmrt {
namespace {

constexpr int kX = 32, kMaxRows = 32;
// halo of a window: 5 for the step; the fields and diagnostics end with u, which needs
// moments up to 4 away (24 instead of 22 own columns and rows of 32: fields of
// 4096^2 790 -> 680 us, diagnostics 1765 -> 1543)
constexpr int edge_of(Pass mode) { return mode == Pass::Step ? 5 : 4; }

__device__ __forceinline__ int wrap(int v, int n) {
    if (v >= 0 && v < n) return v;
    const int r = v % n;
    return r < 0 ? r + n : r;
}
__device__ __forceinline__ void normal_of(float gx, float gy, float& nx, float& ny) {
    const float mag2 = fmaf(gx, gx, gy * gy);
    const float inv = (mag2 >= kNormalTau * kNormalTau) ? rsqrtf(mag2) : 0.0f;
    nx = -gx * inv;
    ny = -gy * inv;
}
// App. B coefficients a_N
__host__ __device__ constexpr float coef(int N) { return N == 1 ? 4.5f : (N == 2 ? -0.9f : 0.1f); }

// ROWS: the window's rows (0: those of the launch); FLAT: a window has the lattice's rows
// and no others (ROWS 0)
template <int ROWS, bool FLAT, bool W, Pass MODE>
__global__ void __launch_bounds__(kX * kMaxRows, 1)
    k_order6(const float* __restrict__ src, float* __restrict__ dst, const StepParams P, FieldOut fo,
             unsigned* __restrict__ flag, double* __restrict__ partials) {
    pdl_begin();
    constexpr int kEdge = edge_of(MODE);
    const int kN = ROWS ? kX * ROWS : static_cast<int>(blockDim.x), H = kN / kX;
    extern __shared__ float sm[];
    const int tx = threadIdx.x % kX, ty = threadIdx.x / kX;
    const int nx = P.nx, ny = P.ny;
    const size_t nodes = static_cast<size_t>(nx) * ny;
    const int xw = static_cast<int>(blockIdx.x) * (kX - 2 * kEdge) - kEdge + tx;
    const int yw = static_cast<int>(blockIdx.y) * (H - 2 * kEdge) - kEdge + ty;
    const int x = wrap(xw, nx), y = FLAT ? ty : W ? yw : wrap(yw, ny);
    const bool in = FLAT || !W || (y >= 0 && y < ny);
    auto inner = [&](int d) { return in && tx >= d && tx < kX - d && (FLAT || (ty >= d && ty < H - d)); };
    const bool own = inner(kEdge) && xw < nx && (FLAT || yw < ny);
    const bool low = W && y == 0, high = W && y == ny - 1;
    float* w = sm + kX + threadIdx.x;  // this node in a field of the window
    constexpr int kChiR = 0, kChiB = 1, kPhi = 2, kGx = 3, kGy = 4, kUx = 5, kUy = 6;
    // window offset of the row y + dy, or of its mirror beyond a wall
    auto row = [&](int dy) {
        int t = y + dy;
        if (W && t < 0) t = -1 - t;
        if (W && t >= ny) t = 2 * ny - 1 - t;
        if (FLAT && !W) t = wrap(t, ny);
        return W || FLAT ? (t - y) * kX : dy * kX;
    };
    auto grad6 = [&](const float* a, float& gx, float& gy) {
        gx = 0.0f;
        gy = 0.0f;
#pragma unroll
        for (int N = 1; N <= 3; ++N) {
            const int rows[3] = {row(-N), 0, row(N)};
#pragma unroll
            for (int i = 1; i < 9; ++i) {
                const float v = a[rows[lcy(i) + 1] + N * lcx(i)];
                if (lcx(i)) gx = fmaf(coef(N) * lw(i) * float(lcx(i)), v, gx);
                if (lcy(i)) gy = fmaf(coef(N) * lw(i) * float(lcy(i)), v, gy);
            }
        }
    };
    // compact derivatives: beyond a wall the node's own row times the field's parity
    const int up = FLAT && !W ? row(1) : high ? 0 : kX, dn = FLAT && !W ? row(-1) : low ? 0 : -kX;
    auto d_x = [&](const float* a, float parity) {
        const float pu = high ? parity : 1.0f, pd = low ? parity : 1.0f;
        return ddx(a[1], a[-1], pu * a[up + 1], pu * a[up - 1], pd * a[dn + 1], pd * a[dn - 1]);
    };
    auto d_y = [&](const float* a, float parity) {
        const float pu = high ? parity : 1.0f, pd = low ? parity : 1.0f;
        return ddy(pu * a[up], pd * a[dn], pu * a[up + 1], pu * a[up - 1], pd * a[dn + 1], pd * a[dn - 1]);
    };

    // ---- moments, colour fractions, Phi'
    float f[9], rr = 1.0f, rb = 1.0f, jx = 0.0f, jy = 0.0f, chr = 0.0f, chb = 0.0f;
    if (in) {
        const unsigned xm = x == 0 ? nx - 1 : x - 1, xp = x == nx - 1 ? 0 : x + 1;
        const unsigned ym = y == 0 ? ny - 1 : y - 1, yp = y == ny - 1 ? 0 : y + 1;
        float fr[9], fb[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            unsigned at = (lcy(i) > 0 ? ym : (lcy(i) < 0 ? yp : static_cast<unsigned>(y))) * nx +
                          (lcx(i) > 0 ? xm : (lcx(i) < 0 ? xp : static_cast<unsigned>(x)));
            int li = i;
            if (W && ((lcy(i) > 0 && low) || (lcy(i) < 0 && high))) {  // half-way bounce-back
                li = lopp(i);
                at = static_cast<unsigned>(y) * nx + x;
            }
            fr[i] = __ldcg(src + nodes * li + at);
            fb[i] = __ldcg(src + nodes * (9 + li) + at);
        }
        rr = ((fr[0] + fr[1]) + (fr[2] + fr[3])) + ((fr[4] + fr[5]) + (fr[6] + fr[7])) + fr[8];
        rb = ((fb[0] + fb[1]) + (fb[2] + fb[3])) + ((fb[4] + fb[5]) + (fb[6] + fb[7])) + fb[8];
#pragma unroll
        for (int i = 0; i < 9; ++i) f[i] = fr[i] + fb[i];
        jx = ((f[1] + f[7]) + f[8]) - ((f[3] + f[5]) + f[4]);
        jy = ((f[1] + f[3]) + f[2]) - ((f[5] + f[7]) + f[6]);
        const float a = rr * P.inv_rho0_r, b = rb * P.inv_rho0_b;
        const float inv = 1.0f / (a + b);
        chr = a * inv;
        chb = b * inv;
        w[kChiR * kN] = chr;
        w[kChiB * kN] = chb;
        w[kPhi * kN] = fmaf(P.phip_r, rr, P.phip_b * rb);
    }
    __syncthreads();
    // ---- grad rho^N on the smaller colour fraction, n-hat
    float gx = 0.0f, gy = 0.0f;
    if (inner(3)) {
        const bool red_minor = chr <= 0.5f;
        grad6(w + (red_minor ? kChiR : kChiB) * kN, gx, gy);
        gx *= red_minor ? 2.0f : -2.0f;
        gy *= red_minor ? 2.0f : -2.0f;
        w[kGx * kN] = gx;
        w[kGy * kN] = gy;
    }
    __syncthreads();
    // ---- K, G, u
    const float rho = rr + rb;
    float Gx = 0.0f, Gy = 0.0f, ux = 0.0f, uy = 0.0f;
    if (inner(4)) {
        float K = P.fixed_K;
        if (P.curvature_mode == 0) {
            // K = div n-hat with n-hat of the neighbours (y odd beyond a wall)
            float nxv[9], nyv[9];
#pragma unroll
            for (int i = 1; i < 9; ++i) {
                const bool mir = W && ((lcy(i) > 0 && high) || (lcy(i) < 0 && low));
                const int o = (lcy(i) > 0 ? up : (lcy(i) < 0 ? dn : 0)) + lcx(i);
                normal_of(w[kGx * kN + o], w[kGy * kN + o], nxv[i], nyv[i]);
                if (W && mir) nyv[i] = -nyv[i];
            }
            K = ddx(nxv[8], nxv[4], nxv[1], nxv[3], nxv[7], nxv[5]) + ddy(nyv[2], nyv[6], nyv[1], nyv[3], nyv[7], nyv[5]);
        }
        const float hk = P.half_sigma * K;
        Gx = fmaf(hk, gx, fmaf(rho, P.gacc_x, P.gvol_x));
        Gy = fmaf(hk, gy, fmaf(rho, P.gacc_y, P.gvol_y));
        ux = fmaf(0.5f, Gx, jx) / rho;
        uy = fmaf(0.5f, Gy, jy) / rho;
        w[kUx * kN] = ux;
        w[kUy * kN] = uy;
    }
    __syncthreads();
    // ---- the node's collision, recolour and store, or its fields
    const size_t at = static_cast<size_t>(y) * nx;
    if (MODE == Pass::Step) {
        if (!own) return;
        if (!isfinite(rho)) atomicOr(flag, 1u);
        float dPx, dPy;
        grad6(w + kPhi * kN, dPx, dPy);
        const float divu = d_x(w + kUx * kN, -1.0f) + d_y(w + kUy * kN, -1.0f);
        const float inv_rho = rcp(rho);
        const float nu = P.visc_mode == 0
                             ? fmaf(0.5f * (P.nu_r - P.nu_b), chr - chb, 0.5f * (P.nu_r + P.nu_b))
                             : P.eta * inv_rho;
        float fp[9];
        collide_increment(f, rr, rb, rho, nu, ux, uy, Gx, Gy, dPx, dPy, divu, P, fp);
        // recolour along e = grad rho^N / |grad rho^N| (Eq. eq_re_color; 0 below kNormalTau)
        const float mag2 = fmaf(gx, gx, gy * gy);
        const float inv = (mag2 >= kNormalTau * kNormalTau) ? rsqrtf(mag2) : 0.0f;
        const float phim = fmaf(P.kphi_r, rr, P.kphi_b * rb) * inv_rho;
        const float sg = P.beta * (rr * rb) * inv_rho * phim * inv;
        store_recoloured_f32(dst + at, x, nodes, fp, rr, rb, inv_rho, sg * gx, sg * gy);
    } else if (MODE == Pass::Fields) {
        if (!own) return;
        const size_t o = at + x;
        if (fo.rho_r) fo.rho_r[o] = rr;
        if (fo.rho_b) fo.rho_b[o] = rb;
        if (fo.ux) fo.ux[o] = ux;
        if (fo.uy) fo.uy[o] = uy;
        if (fo.p) fo.p[o] = fmaf(P.cs2_r, rr, P.cs2_b * rb);
    } else {
        // FP64 partial diagnostics of the CTA (slot 4 is a maximum): a warp per two sums and
        // one for the fastest node, a lane per column, over values left in the place of
        // fields that are read no more.  A warp's FP64 instruction takes the SM 16 cycles:
        // six FP64 shuffle reductions in every warp took two thirds of the pass (4096^2
        // 3790 us, this 1765)
        const bool counts = own && isfinite(rho);
        const float part[6] = {rr, rb, jx, jy, ux, uy};
#pragma unroll
        for (int j = 0; j < 6; ++j) w[(j < 4 ? j : j + 1) * kN] = counts ? part[j] : 0.0f;
        const int bad = __syncthreads_count(own && !counts);
        double* out = partials + (static_cast<size_t>(blockIdx.y) * gridDim.x + blockIdx.x) * kDiagSlots;
        const int first = FLAT ? 0 : kEdge;
        for (int q = ty; q < 3; q += H) {
            const float *a = sm + kX + (q < 2 ? 2 * q : kUx) * kN + tx, *b = a + kN;
            double v = 0.0, v2 = 0.0;
            if (q < 2) {
                Sum3 sum;
                for (int k = first; k < H - first; ++k) {
                    const float c = a[k * kX], d = b[k * kX];
                    if (fmaxf(fabsf(c), fabsf(d)) < 1e30f) {
                        sum.add(c, d);
                    } else {
                        v += c;
                        v2 += d;
                    }
                }
                sum.take(v, v2);
            } else {
                Fastest fastest;
                for (int k = first; k < H - first; ++k) fastest.add(a[k * kX], b[k * kX], v);
                fastest.take(v);
            }
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) {
                const double u = __shfl_down_sync(0xffffffffu, v, off);
                v = q == 2 ? fmax(v, u) : v + u;
                if (q < 2) v2 += __shfl_down_sync(0xffffffffu, v2, off);
            }
            if (tx == 0) {
                out[2 * q] = v;
                out[2 * q + 1] = q < 2 ? v2 : static_cast<double>(bad);
            }
        }
    }
}

// Lattices of at most 32 rows are one window high, without halo rows: the row beyond
// an edge, periodic or mirrored, is a row of the window.  150000 x 4: 30 us per step
// with 4 window rows, 148 with 32 of which 22 own (45 as plane passes); 20000 x 24: 30
// against 48 (35).
bool flat6(int ny) { return ny <= kMaxRows; }

dim3 grid6(int nx, int ny, int H, int edge) {
    const int tx = kX - 2 * edge, ty = H - 2 * edge;
    return dim3(static_cast<unsigned>((nx + tx - 1) / tx), flat6(ny) ? 1u : static_cast<unsigned>((ny + ty - 1) / ty));
}

// Window rows: the lattice's where it is flat; else 16 (two CTAs per SM) while that is
// at most two windows per SM, else 32, or those of 17 to 31 of a periodic lattice that
// save at least 4 % of the rows computed (rows known only at the launch cost 1 to 2 %;
// halo rows beyond a wall are idle anyway).  20000 x 33: 56 us per step with 32 rows,
// 52 with 27.
int rows6(const StepParams& P, int edge) {
    if (flat6(P.ny)) return P.ny;
    const dim3 g = grid6(P.nx, P.ny, 16, edge);
    if (static_cast<long>(g.x) * g.y <= 304) return 16;
    int best = kMaxRows;
    auto computed = [&](int H) { return static_cast<long>((P.ny + H - 2 * edge - 1) / (H - 2 * edge)) * H; };
    for (int H = kMaxRows - 1; H > 16 && !P.wall_y; --H)
        if (computed(H) < computed(best) && computed(H) * 100 <= computed(kMaxRows) * 96) best = H;
    return best;
}

template <Pass MODE>
cudaError_t launch6(const float* src, float* dst, const StepParams& P, FieldOut fo, unsigned* flag, double* partials,
                    cudaStream_t s) {
    const int H = rows6(P, edge_of(MODE));
    const dim3 g = grid6(P.nx, P.ny, H, edge_of(MODE));
    auto go = [&](auto k) {
        return launch_pdl(k, g, dim3(kX * H), (7 * kX * H + 2 * kX) * sizeof(float), s, src, dst, P, fo, flag, partials);
    };
    if (flat6(P.ny)) return P.wall_y ? go(&k_order6<0, true, true, MODE>) : go(&k_order6<0, true, false, MODE>);
    if (H == 16) return P.wall_y ? go(&k_order6<16, false, true, MODE>) : go(&k_order6<16, false, false, MODE>);
    if (H == 32) return P.wall_y ? go(&k_order6<32, false, true, MODE>) : go(&k_order6<32, false, false, MODE>);
    return go(&k_order6<0, false, false, MODE>);
}

}  // namespace

cudaError_t launch_step6(const float* src, float* dst, const StepParams& P, unsigned* flag, cudaStream_t s) {
    return launch6<Pass::Step>(src, dst, P, FieldOut{}, flag, nullptr, s);
}
cudaError_t launch_fields6(const float* src, const StepParams& P, FieldOut out, cudaStream_t s) {
    return launch6<Pass::Fields>(src, nullptr, P, out, nullptr, nullptr, s);
}
int diag_blocks6(const StepParams& P) {
    const dim3 g = grid6(P.nx, P.ny, rows6(P, edge_of(Pass::Diag)), edge_of(Pass::Diag));
    return static_cast<int>(g.x * g.y);
}
cudaError_t launch_diag6(const float* src, const StepParams& P, double* partials, cudaStream_t s) {
    return launch6<Pass::Diag>(src, nullptr, P, FieldOut{}, nullptr, partials, s);
}

}  // namespace cmrt
