// Fused chromodynamic MRT step (arXiv 2005.04642, Sec. 2, Sec. 3, App. A)
// as one row-marching kernel for sm_103a.
//
// Data layout in HBM: the state is the post-collision (pre-streaming)
// populations P_{t-1}.  With FP32 storage they are 18 planes
// float[18][ny][nx] (red links 0..8, then blue links 0..8).  With 16-bit
// storage (FP16 or BF16) a node keeps its two colour densities and its two
// rest populations in FP32 and twelve 16-bit (red, blue) pairs: four
// reference dipoles -- the equilibrium's velocity term and the recolour's
// segregation term -- and the deviations d_{C,i} = C_i - rho_C psi_i -/+ D_C
// of the eight moving links from a reference that scales with the node's own
// colour density: planes 0 and 1 are float2[ny][nx] (rho_R, rho_B) and
// (R_0, B_0), planes 2..13 16-bit pairs.  The rest populations are the
// remainder of the densities after the decoded moving links, so a record
// decodes to populations summing to rho_C.
// One launch gathers the pre-collision populations f(t) = stream(P_{t-1})
// on the fly ("pull"), performs the whole per-node update and writes P_t to
// the other buffer at the node itself, so every HBM access is coalesced:
// 72 B (FP32) or 64 B (16-bit) read and as much written per node.
//
// A CTA owns a strip of columns (a window of 128 less 4 halo columns on each
// side, one thread per window column) and marches down a segment of rows,
// which stream into shared memory with 16-byte cp.async copies.  Each
// iteration runs a wavefront of four stages on consecutive rows:
//   A (row r)      gather f, colour moments, colour fractions       (tile + 3)
//   B (row r - 1)  grad rho^N and n-hat with the compact stencil    (tile + 2)
//   C (row r - 2)  K = div n-hat, force G, force-adjusted u, Phi'   (tile + 1)
//   D (row r - 4)  grad Phi', div u, C_ab, MRT collision in moment
//                  space, reconstruction, recolour, store           (tile)
// so the stencil chain of radius 3 costs only the recomputation of the halo
// moments and never re-reads HBM.
//
// The collision is written in increment form, f+ = f + M^{-1} dm with
// dm = Lambda (m^(0) - m) + S (App. A, Eq. 38 minus m): the increments are
// small, so FP32 rounding stays at the level of population storage.  The
// reconstruction M^{-1} dm is grouped by the parity of each column k^(p)
// under c -> -c, which the k vectors of App. A have by construction.
#pragma once

#include <atomic>
#include <type_traits>

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "cmrt_device.cuh"

namespace cmrt {
namespace {

constexpr int kPlanes = 18;
// The reconstruction below relies on these symmetries of App. A's k vectors.
static_assert(kinv(4, 3) == kinv(8, 3) && kinv(4, 4) == kinv(8, 4) && kinv(4, 6) == kinv(8, 6), "even x");
static_assert(kinv(4, 1) == -kinv(8, 1) && kinv(4, 7) == -kinv(8, 7), "odd x");
static_assert(kinv(6, 3) == kinv(2, 3) && kinv(6, 4) == kinv(2, 4) && kinv(6, 6) == kinv(2, 6), "even y");
static_assert(kinv(6, 2) == -kinv(2, 2) && kinv(6, 8) == -kinv(2, 8), "odd y");
static_assert(kinv(2, 3) == kinv(8, 4) && kinv(2, 4) == kinv(8, 3) && kinv(2, 2) == kinv(8, 1) &&
              kinv(2, 8) == kinv(8, 7), "x <-> y");
static_assert(kinv(1, 3) == kinv(1, 4) && kinv(1, 1) == kinv(1, 2) && kinv(1, 7) == kinv(1, 8), "diagonal");
static_assert(kinv(8, 2) == 0.f && kinv(8, 5) == 0.f && kinv(8, 8) == 0.f && kinv(0, 1) == 0.f &&
              kinv(0, 5) == 0.f && kinv(0, 7) == 0.f, "zeros");

__device__ __forceinline__ void cp_async16(unsigned smem_addr, const void* gmem) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem_addr), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async8(unsigned smem_addr, const void* gmem) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(smem_addr), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async4(unsigned smem_addr, const void* gmem) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(smem_addr), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

__device__ __forceinline__ int wrap(int v, int n) {
    int r = v % n;
    return r < 0 ? r + n : r;
}

// (sum over links of r, of b), pairwise, as packed FP32x2 adds (one instruction per pair)
__device__ __forceinline__ float2 sum9x2(const float (&r)[9], const float (&b)[9]) {
    float2 v[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) v[i] = make_float2(r[i], b[i]);
    const float2 a = __fadd2_rn(__fadd2_rn(v[0], v[1]), __fadd2_rn(v[2], v[3]));
    const float2 c = __fadd2_rn(__fadd2_rn(v[4], v[5]), __fadd2_rn(v[6], v[7]));
    return __fadd2_rn(__fadd2_rn(a, c), v[8]);
}

// ---------------------------------------------------------------------------
// The 16-bit record: how a node is decoded, and encoded by the step's last stage.
// (How the march copies rows of either storage and hands them to stage A: MarchF32
// and March16.)
// ---------------------------------------------------------------------------

// 16-bit deviations (H = __half2 or __nv_bfloat162).
//
// Record of a node: two float2 planes -- the colour densities (rho_R,
// rho_B) and the rest populations (R_0, B_0) -- then twelve planes of 16-bit
// (red, blue) pairs -- four reference dipoles D_0..D_3, then the deviations
// d_i of the moving links i = 1..8 -- decoded as
//   C_i = rho_C psi_i + (+/-) D_C,dip(i) + d_C,i / 2^k      (i >= 1)
// (dip_index, dip_neg).  psi_i are the reference weights of the axis and
// diagonal links (weights()), of the shape that the lowest bit of D_0's red
// half selects (the record's flag).  The step stores as dipoles (dipoles16) the
// equilibrium's velocity term, with the node's post-collision velocity, and
// the recolour's segregation term (Eq. eq_re_color), so that its deviations
// are only the non-equilibrium and second-order parts of the populations:
// tens of times smaller than their deviations from rho_C psi_i, and so is
// their 16-bit rounding.  The dipoles are reference values, stored rounded
// and used as stored: their rounding only moves a little into the
// deviations.  The rest populations are the remainder of rho_C after the
// decoded moving links, so that a record decodes to populations summing to
// rho_C.  Any pair of population sets is representable.
template <class H>
struct Layout16 {
    static constexpr int kPairPlanes = 12;  // four dipoles, eight deviations
    static constexpr size_t node_bytes() { return 16 + kPairPlanes * 4; }

    __device__ __forceinline__ static float2 to2(H v);
    __device__ __forceinline__ static H from2(float a, float b);
    __device__ __forceinline__ static H from2x(float2 v) { return from2(v.x, v.y); }

    // Reference weights (psi_a, psi_d) of a node's axis and diagonal links, as
    // (red, blue) pairs.  psi_a: precision_reference 0 phi_i of Eq. eq_phi at
    // the node's own mixture, ((1 - alpha_R) rho_R + (1 - alpha_B) rho_B) /
    // (5 rho) rounded to a multiple of 2^-24; otherwise per-colour constants
    // (psi_r, psi_b).  Two shapes, chosen per record by its flag (the lowest
    // bit of D_0's red half): psi_d = psi_a / 4 (flag 0), the equilibrium's
    // shape, whose ghost moment N is the equilibrium one; or (flag 1) the rest
    // state with the same mass and energy and N = 0, which is what the
    // collision leaves where N relaxes to 0 (ghost_N_mode 1): with Dellar's
    // ghost weights g = (1, -2, 4) for the rest, axis and diagonal links,
    // psi_a' = psi_a / 2 + 1/18 and psi_d' = psi_a / 2 - 1/36.  Any choice
    // decodes correctly; a reference far from the populations only makes the
    // deviations, and their 16-bit rounding, larger.
    __device__ __forceinline__ static void weights(float rr, float rb, float inv_rho, bool nfree,
                                                   const StepParams& P, float2& wa, float2& wd) {
        float2 pa;
        if (P.precision_reference == 0) {
            float s5 = fmaf(P.mix_r, rr, P.mix_b * rb) * inv_rho;
            s5 = fminf(fmaxf(s5, 0.0f), 0.25f);
            const float q = __fsub_rn(__fadd_rn(s5, 0.5f), 0.5f);  // a multiple of 2^-24
            pa = make_float2(q, q);
        } else {
            pa = make_float2(P.psi_r[1], P.psi_b[1]);
        }
        // one form for both shapes: pa * s + c, with (s, c) = (1, 0) and (1/4, 0)
        // exact for the equilibrium's
        const float sa = nfree ? 0.5f : 1.0f, ca = nfree ? 1.0f / 18.0f : 0.0f;
        const float sd = nfree ? 0.5f : 0.25f, cd = nfree ? -1.0f / 36.0f : 0.0f;
        wa = __ffma2_rn(pa, make_float2(sa, sa), make_float2(ca, ca));
        wd = __ffma2_rn(pa, make_float2(sd, sd), make_float2(cd, cd));
    }

    // link class of link i >= 1: axis (even i) or diagonal (odd i)
    __device__ __forceinline__ static constexpr bool diag(int i) { return (i & 1) != 0; }

    // The populations (red, blue) of a record: its densities, rest populations
    // and twelve pairs.
    __device__ __forceinline__ static void decode(float2 rho, float2 rest, const H (&raw)[12], const StepParams& P,
                                                  float2 (&c)[9]) {
        float2 wa, wd;
        weights(rho.x, rho.y, rcp(rho.x + rho.y), (*reinterpret_cast<const unsigned*>(&raw[0]) & 1u) != 0, P, wa, wd);
        const float2 refa = __fmul2_rn(rho, wa), refd = __fmul2_rn(rho, wd);
        const float2 un2 = make_float2(P.dev_unscale, P.dev_unscale), m1 = make_float2(-1.0f, -1.0f);
        c[0] = rest;
#pragma unroll
        for (int i = 1; i < 9; ++i) {
            // reference pair plus the stored deviation times 2^-k (exact), rounded once; then the dipole
            c[i] = __ffma2_rn(to2(raw[3 + i]), un2, diag(i) ? refd : refa);
            const float2 D = to2(raw[dip_index(i)]);
            c[i] = dip_neg(i) ? __ffma2_rn(D, m1, c[i]) : __fadd2_rn(c[i], D);
        }
    }

    // The populations of the node in column x of the row that starts at node `row`.
    __device__ __forceinline__ static void load(const char* state, size_t nodes, size_t row, unsigned x,
                                                const StepParams& P, float2 (&c)[9]) {
        const float2* own = reinterpret_cast<const float2*>(state) + row;
        const unsigned* pairs = reinterpret_cast<const unsigned*>(state + nodes * 16) + row;
        const float2 rho = __ldcg(own + x), rest = __ldcg(own + nodes + x);
        H raw[12];
#pragma unroll
        for (int j = 0; j < 12; ++j) {
            const unsigned v = __ldcg(pairs + j * nodes + x);
            raw[j] = *reinterpret_cast<const H*>(&v);
        }
        decode(rho, rest, raw, P, c);
    }

    // The node is column x of the row that starts at node `row`.
    __device__ __forceinline__ static void store(char* dst, size_t nodes, size_t row, unsigned x,
                                                 const float (&fp)[9], float rr, float rb, float inv_rho, float sx,
                                                 float sy, float ux, float uy, const StepParams& P) {
        // The recoloured pair of link i is (rho_C / rho) f+_i +/- s_i (Eq.
        // eq_re_color); the record keeps it minus the dipole and the reference,
        // scaled by 2^k (dev_scale) before rounding to 16 bits (a power-of-two
        // factor commutes exactly with FP32 rounding).
        const float S = P.dev_scale;
        H* pairs = reinterpret_cast<H*>(dst + nodes * 16) + row;
        float2 D[4];
        dipoles16(rr, rb, ux, uy, sx, sy, D);
        // the reference flag: N-free shape where the collision relaxes N to 0
        const bool nfree = P.ghost_N_mode == 1;
        float2 Dq[4];  // as stored, and as the decoder will use them
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            H h = from2x(D[j]);
            if (j == 0) {
                // the flag replaces the lowest bit of D_0's red half: a reference
                // value, so the change moves into the deviations exactly
                unsigned u = *reinterpret_cast<const unsigned*>(&h);
                u = (u & ~1u) | (nfree ? 1u : 0u);
                h = *reinterpret_cast<const H*>(&u);
            }
            (pairs + j * nodes)[x] = h;
            Dq[j] = to2(h);
        }
        float seg[9];
        segregation(sx * S, sy * S, seg);
        const float2 rho2 = make_float2(rr, rb);
        float2 wa, wd;
        weights(rr, rb, inv_rho, nfree, P, wa, wd);
        const float2 refa = __fmul2_rn(rho2, wa);  // the decoder's reference pairs
        const float2 refd = __fmul2_rn(rho2, wd);
        const float ar = rr * inv_rho * S, ab = rb * inv_rho * S;
        const float2 mrho = make_float2(-rr * S, -rb * S);
        const float2 mS = make_float2(-S, -S), pS = make_float2(S, S), m1 = make_float2(-1.0f, -1.0f);
        const float2 un2 = make_float2(P.dev_unscale, P.dev_unscale);
        // The rest populations are what is left of rho_R and rho_B after the
        // moving links as the decoder will see them (decode(), bit for bit), so
        // that every record decodes to exactly its colour densities: colour mass
        // is conserved through the storage to the rounding of that sum.
        float2 sum = make_float2(0.0f, 0.0f);
#pragma unroll
        for (int i = 1; i < 9; ++i) {
            // two scalar FMAs: packed, the operands' copies into pairs cost more than it saves
            float2 C = make_float2(__fmaf_rn(ar, fp[i], seg[i]), __fmaf_rn(ab, fp[i], -seg[i]));
            const float2 Dj = Dq[dip_index(i)];
            C = __ffma2_rn(Dj, dip_neg(i) ? pS : mS, C);
            const H h = from2x(__ffma2_rn(mrho, diag(i) ? wd : wa, C));
            (pairs + (3 + i) * nodes)[x] = h;
            const float2 d = to2(h);
            float2 c = __ffma2_rn(d, un2, diag(i) ? refd : refa);
            c = dip_neg(i) ? __ffma2_rn(Dj, m1, c) : __fadd2_rn(c, Dj);
            sum = __fadd2_rn(sum, c);
        }
        float2* own = reinterpret_cast<float2*>(dst) + row;
        own[x] = rho2;
        (own + nodes)[x] = __ffma2_rn(sum, m1, rho2);
    }
};

template <>
__device__ __forceinline__ float2 Layout16<__half2>::to2(__half2 v) { return __half22float2(v); }
template <>
__device__ __forceinline__ __half2 Layout16<__half2>::from2(float a, float b) { return __floats2half2_rn(a, b); }
template <>
__device__ __forceinline__ float2 Layout16<__nv_bfloat162>::to2(__nv_bfloat162 v) { return __bfloat1622float2(v); }
template <>
__device__ __forceinline__ __nv_bfloat162 Layout16<__nv_bfloat162>::from2(float a, float b) {
    return __floats2bfloat162_rn(a, b);
}

// Diagnostics accumulators of one thread (Pass::Diag).
struct DiagAcc {
    double r = 0.0, b = 0.0, jx = 0.0, jy = 0.0, u2 = 0.0, bad = 0.0;
};

// Local kinematic viscosity (Sec. 2: nu(rho^N) = (2 / lambda_3 - 1) / 6), rho^N by Eq. equ_rhoN_def.
__device__ __forceinline__ float node_viscosity(float rr, float rb, float inv_rho, const StepParams& P) {
    if (P.visc_mode != 0) return P.eta * inv_rho;
    const float ra = rr * P.inv_rho0_r, ba = rb * P.inv_rho0_b;
    const float rn = (ra - ba) * rcp(ra + ba);
    return fmaf(0.5f * (P.nu_r - P.nu_b), rn, 0.5f * (P.nu_r + P.nu_b));
}

// ---------------------------------------------------------------------------
// The march: the row pipeline of one tile.
//
// A CTA of 128 threads, one per window column, runs all four stages of every
// row itself; four such CTAs (16 warps) share an SM.  Row iteration k
// (r = y0 - 3 + k) runs, with one barrier before each group,
//   D (row r - 4), A (row r) | B (row r - 1) | C (row r - 2).
// What bounds it: HBM.  144 B per node are the algorithm's; to stream them an
// SM has to keep 40 KB in flight and to issue few instructions per node, and
// both come from where the data between the stages lives:
// - Every population is gathered exactly once, by stage A.  With FP32 storage a
//   slot of shared memory holds what gather row r needs (plane q from row
//   r - c_y(q)), so a row is dead as soon as A has read it and three slots (one
//   in use, two in flight) serve where a ring of whole rows kept for stage D
//   took nine.
// - Stage D gets f, rho_R and rho_B of its row from registers, where A left
//   them four iterations before, instead of gathering and summing the eighteen
//   populations again.
// - The smaller shared memory (42 KB against 114 KB) lets four CTAs of four
//   warps stand on an SM: 512 columns in flight, against 256 with two CTAs of
//   eight warps that split the stages between them, and each warp has the whole
//   work of a row to overlap the others' barriers.
// - 630 thread instructions per node, 834 with FP16 storage (836 and 1140 where two
//   groups of warps split the stages).
// Measured at 8192^2 (drops, FP32): 1982 us per step before (33.9 GLUPS,
// 4.9 TB/s), 1643 us now (40.9 GLUPS, 5.9 TB/s, 87 % of the measured copy);
// 2048^2 143 -> 120 us; FP16 8192^2 2488 -> 1893 us, BF16 2614 -> 2001 us (bound
// by issue: 72 % of the slots).  Two and four slots: 1851 and 1678 us.  Three
// CTAs per SM (168 registers): 1698 us.  256-column windows (two CTAs of eight
// warps) 1930 us: fewer barrier domains to overlap.  The loop is unrolled
// twice: four times saves the moves of the register FIFO (13 per row) but the
// code no longer fits the instruction caches (FP16 1980 us, with walls 2190).
// ---------------------------------------------------------------------------
// resident CTAs per SM with W window columns (and threads): 16 warps of 128
// registers, or 15 of the 96-column window
template <int W>
constexpr int march_ctas() { return 512 / W; }
constexpr int kMarchRows = 28;  // stage rings, four rows each: chi_R, chi_B, Phi', n-hat x, y, u x, y

// A tile: the strip of own columns from x0 of n rows from y0 of a lattice.  A
// kernel of one lattice has it in its parameters; the batched kernel keeps it
// in shared memory (with the member's StepParams) and the march reads each
// value where it needs it, rather than hold some twenty registers per thread.
struct Tile {
    const char* src;
    char* dst;
    unsigned* flag;
    size_t nodes;
    int nx, ny, wall, x0, y0, n;
    Tile() = default;
    __device__ __forceinline__ Tile(const char* s, char* d, unsigned* f, const StepParams& P, int x0_, int y0_, int rows)
        : src(s), dst(d), flag(f), nodes(static_cast<size_t>(P.nx) * P.ny), nx(P.nx), ny(P.ny), wall(P.wall_y), x0(x0_),
          y0(y0_), n(min(rows, P.ny - y0_)) {}
    __device__ __forceinline__ size_t row_bytes() const { return static_cast<size_t>(nx) * 4; }
};

template <int C>
using Const = std::integral_constant<int, C>;

// This thread's share of the copy of a gather row: with VEC (nx a multiple of
// 4) 16-byte chunks, warp w copying planes w, w + 4, ... and a lane four
// columns; otherwise its own column of every plane.  PRE: the populations
// already lie where they are needed (the public layout).
template <int W, bool VEC, bool WALLS, bool PRE>
struct MarchCopy {
    static constexpr int kN = VEC ? (kPlanes + 3) / 4 : 1;
    const char* ptr[kN];  // column of plane q in row -c_y(q)
    __device__ __forceinline__ static int plane_of(int m) { return static_cast<int>(threadIdx.x) / (W / 4) + 4 * m; }
    // c_y of the link of plane q
    __device__ __forceinline__ static int plane_cy(int q) {
        const int l = q >= 9 ? q - 9 : q;
        return PRE ? 0 : (l >= 5 && l <= 7 ? -1 : (l >= 1 && l <= 3 ? 1 : 0));
    }
    __device__ __forceinline__ void init(const Tile& T) {
        if (VEC) {
            const int col = wrap(T.x0 - kHalo + static_cast<int>(threadIdx.x) % (W / 4) * 4, T.nx);
#pragma unroll
            for (int m = 0; m < kN; ++m)
                ptr[m] = T.src + T.nodes * 4 * plane_of(m) + static_cast<size_t>(col) * 4 -
                         static_cast<ptrdiff_t>(T.row_bytes()) * plane_cy(plane_of(m));
        } else {
            ptr[0] = T.src + static_cast<size_t>(wrap(T.x0 - kHalo + static_cast<int>(threadIdx.x), T.nx)) * 4;
        }
    }
    // (WALLS: a lattice that may have walls, T.wall whether it has)
    // byte offset from plane q's row 0 to the row that gather row r takes from it
    __device__ __forceinline__ static ptrdiff_t row_off(const Tile& T, int r, int cy) {
        int g = r - cy;
        if (g < 0 || g >= T.ny) {
            // half-way bounce-back: the node's own row of the opposite link's plane
            if (WALLS && T.wall) return static_cast<ptrdiff_t>(T.nodes) * (cy > 0 ? 16 : -16) +
                                        static_cast<ptrdiff_t>(T.row_bytes()) * r;
            g = wrap(g, T.ny);
        }
        return static_cast<ptrdiff_t>(T.row_bytes()) * g;
    }
    // the populations of gather row r into a slot: plane q from row r - c_y(q)
    __device__ __forceinline__ void issue(const Tile& T, unsigned slot_addr, int r) const {
        const ptrdiff_t row = T.row_bytes();
        if (VEC) {
            const unsigned d = slot_addr + threadIdx.x * 16;
            if (r >= 1 && r <= T.ny - 2) {
                const ptrdiff_t o = row * r;
#pragma unroll
                for (int m = 0; m < kN; ++m)
                    if (4 * m + 3 < kPlanes || plane_of(m) < kPlanes) cp_async16(d + m * 16 * W, ptr[m] + o);
            } else {
#pragma unroll
                for (int m = 0; m < kN; ++m) {
                    const int q = plane_of(m), cy = plane_cy(q);
                    if (q < kPlanes) cp_async16(d + m * 16 * W, ptr[m] + (row_off(T, r, cy) + row * cy));
                }
            }
        } else {
            const unsigned d = slot_addr + threadIdx.x * 4;
            const ptrdiff_t om = PRE ? 0 : row_off(T, r, -1), oz = row_off(T, r, 0), op = PRE ? 0 : row_off(T, r, 1);
#pragma unroll
            for (int q = 0; q < kPlanes; ++q) {
                const int cy = PRE ? 0 : lcy(q % 9);
                cp_async4(d + q * W * 4,
                          ptr[0] + (static_cast<ptrdiff_t>(T.nodes) * 4 * q + (cy > 0 ? op : (cy < 0 ? om : oz))));
            }
        }
    }
};

// FP32 storage: a slot holds one gather row, read by stage A alone.
template <int W_>
struct MarchF32 {
    static constexpr int W = W_;
    static constexpr bool kDecode = false;
    static constexpr int kSlots = 3;                     // one in use, two in flight
    static constexpr int kSlotBytes = kPlanes * W * 4;
    static constexpr int kBytes = kSlots * kSlotBytes + kMarchRows * W * 4;
    static constexpr int kLead = 0;
    template <bool VEC, bool WALLS, bool PRE>
    using Copy = MarchCopy<W, VEC, WALLS, PRE>;
};

// 16-bit storage (the record of Layout16): rows of records are copied as they
// lie, and each is decoded once, by the thread of its own column, into FP32
// populations in shared memory (a (red, blue) pair per column and link), from
// where stage A gathers as in FP32.
// Decoding inside the gather, as the earlier two-group form did, decodes every
// record twice (stages A and D) and each of its links with its neighbour's
// reference.  A decoded plane keeps the rows its gather still needs: four of
// the links with c_y = 1 (rows r - 1 .. r + 2 of iteration r; four for a
// compile-time slot), two of the others (two of c_y = -1 only for a wall).
template <class H, int W_>
struct March16 {
    static constexpr int W = W_;
    using Record = Layout16<H>;
    static constexpr bool kDecode = true;
    static constexpr int kSlots = 2;                     // rows of records: one in use, one in flight
    static constexpr int kRefBytes = W * 8;           // (rho_R, rho_B), then (R_0, B_0), float2 per column
    static constexpr int kPairOff = 2 * kRefBytes;
    static constexpr int kSlotBytes = kPairOff + 12 * W * 4;
    static constexpr int kDecBytes = 24 * W * 8;         // decoded rows, a (red, blue) pair per column
    static constexpr int kBytes = kSlots * kSlotBytes + kDecBytes + kMarchRows * W * 4;
    static constexpr int kLead = 3;                      // iterations that only decode
    // first decoded row of link i
    __device__ __forceinline__ static constexpr int dec_row(int i) {
        return lcy(i) > 0 ? 4 * (i - 1) : (lcy(i) < 0 ? 18 + 2 * (i - 5) : 12 + 2 * (i == 0 ? 0 : (i == 4 ? 1 : 2)));
    }

    // This thread's share of the copy of a row of records: with VEC four
    // 16-byte chunks, otherwise its own column.
    template <bool VEC, bool WALLS, bool PRE>
    struct Copy {
        const char* two;   // this thread's chunk or column of the densities or rest populations, row 0
        const char* pair;  // of its first pair plane
        unsigned x;        // without VEC: its column
        __device__ __forceinline__ void init(const Tile& T) {
            const int t = threadIdx.x;
            if (VEC) {
                two = T.src + (t >= W / 2 ? T.nodes * 8 : 0) +
                      static_cast<size_t>(wrap(T.x0 - kHalo + t % (W / 2) * 2, T.nx)) * 8;
                pair = T.src + T.nodes * 16 + static_cast<size_t>(t / (W / 4)) * T.nodes * 4 +
                       static_cast<size_t>(wrap(T.x0 - kHalo + t % (W / 4) * 4, T.nx)) * 4;
            } else {
                x = wrap(T.x0 - kHalo + t, T.nx);
            }
        }
        __device__ __forceinline__ void issue(const Tile& T, unsigned slot, int r) const {
            const int g = r >= 0 && r < T.ny ? r : wrap(r, T.ny);
            const size_t o = static_cast<size_t>(T.nx) * g, nodes = T.nodes;
            const unsigned t = threadIdx.x;
            if (VEC) {
                cp_async16(slot + t * 16, two + o * 8);
#pragma unroll
                for (int m = 0; m < 3; ++m) cp_async16(slot + kPairOff + (t + m * W) * 16, pair + (o + 4 * m * nodes) * 4);
            } else {
                const char* row = T.src + o * 8;
                cp_async8(slot + t * 8, row + x * 8u);
                cp_async8(slot + kRefBytes + t * 8, row + nodes * 8 + x * 8u);
                row = T.src + nodes * 16 + o * 4;
#pragma unroll
                for (int q = 0; q < 12; ++q) cp_async4(slot + kPairOff + (q * W + t) * 4, row + q * nodes * 4 + x * 4u);
            }
        }
    };

    // The record of column t in a slot into the decoded rows (dec: column t),
    // the links with c_y = 1 at s4 pairs from their first row, the others at s2.
    __device__ __forceinline__ static void decode(const char* slot, int t, float2* dec, int s4, int s2,
                                                  const StepParams& P) {
        const float2 rho = reinterpret_cast<const float2*>(slot)[t];
        const float2 rest = reinterpret_cast<const float2*>(slot + kRefBytes)[t];
        const H* pairs = reinterpret_cast<const H*>(slot + kPairOff) + t;
        H raw[12];
#pragma unroll
        for (int j = 0; j < 12; ++j) raw[j] = pairs[j * W];
        float2 c[9];
        Record::decode(rho, rest, raw, P, c);
#pragma unroll
        for (int i = 0; i < 9; ++i) dec[dec_row(i) * W + (lcy(i) > 0 ? s4 : s2)] = c[i];
    }
};
// 1 KB reserved per CTA, and up to 512 B static in the batched kernel
static_assert(march_ctas<128>() * (MarchF32<128>::kBytes + 1536) <= 228 * 1024, "resident FP32 march CTAs");
static_assert(march_ctas<128>() * (March16<__half2, 128>::kBytes + 1536) <= 228 * 1024, "resident 16-bit march CTAs");
static_assert(march_ctas<96>() * (March16<__half2, 96>::kBytes + 1536) <= 228 * 1024, "resident 96-column CTAs");

// The strip [x0, x0 + 120) of rows [y0, y0 + rows).  Window columns whose
// neighbours lie outside the window hold garbage, one more on each side after
// every stage; the four halo columns keep it off the owned ones.  Leaves no
// copy in flight.
//
// Ring slots: row r - j of iteration k is in slot (k - j) mod 4 of every stage
// ring.  chi is read down to row r - 2 by B, n-hat to r - 3 by C (and
// r - 4 by D, the own column), u and Phi' to r - 5 by D, each at least one
// barrier before its slot is written again.  Beyond a wall a stage writes the
// mirrored row together with the wall row, into the slot of the row four
// away, which no later stage reads any more.
template <class L, bool VEC, bool WALLS, Pass MODE, bool PRE>
__device__ __forceinline__ void march_tile(char* __restrict__ smem, const Tile& T, const StepParams& P,
                                           const FieldOut& fo, DiagAcc& acc) {
    constexpr bool kStep = MODE == Pass::Step || MODE == Pass::StepFields;
    constexpr int W = L::W;
    constexpr int kLead = L::kLead;
    const int t = static_cast<int>(threadIdx.x);
    const int rows = T.n;
    const int iters = rows + 7 + kLead;
    const int r_first = T.y0 - 3 - kLead;
    const unsigned pop_addr = static_cast<unsigned>(__cvta_generic_to_shared(smem));
    // this thread's column of the decoded rows (16-bit storage) and of the stage rings
    float2* dec = reinterpret_cast<float2*>(smem + L::kSlots * L::kSlotBytes) + t;
    float* ring = reinterpret_cast<float*>(smem + L::kBytes) - kMarchRows * W + t;
    auto row_ok = [&](int r) { return !WALLS || !T.wall || (r >= 0 && r < T.ny); };
    auto at_low = [&](int r) { return WALLS && T.wall && r == 0; };
    auto at_high = [&](int r) { return WALLS && T.wall && r == T.ny - 1; };
    __shared__ float density[MODE == Pass::Fields ? 2 * W : 1];  // fields: rho_R, rho_B of D's row
    const int gx_own = T.x0 + t - kHalo;
    const bool own_col = t >= kHalo && t < W - kHalo && gx_own < T.nx;
    // iteration k handles own row k - kLead - 3 - d at a stage d rows behind stage A
    auto owned = [&](int k, int d) {
        const int j = k - kLead - 3 - d;
        return MODE == Pass::StepFields && own_col && j >= 0 && j < rows;
    };
    // (a plane's row address is common to the CTA)
    auto fwd = [&](int plane, int r) -> float& {
        return (fo.fwd + static_cast<size_t>(plane) * T.nodes + static_cast<size_t>(r) * T.nx)[static_cast<unsigned>(gx_own)];
    };
    // ring rows (column t): field f of the row in slot c; slots 0, 1 and 2, 3 of an
    // iteration trade places every two iterations
    int half = 0;
    auto R = [&](int f, int c) { return ring + ((f * 4 + (c & 1)) * W + ((c & 2) ? 2 * W - half : half)); };
    constexpr int kChiR = 0, kChiB = 1, kPhi = 2, kNx = 3, kNy = 4, kUx = 5, kUy = 6;
    auto dx = [&](int f, int n, int m, int s) {
        const float *a = R(f, n), *b = R(f, m), *c = R(f, s);
        return ddx(b[1], b[-1], a[1], a[-1], c[1], c[-1]);
    };
    auto dy = [&](int f, int n, int s) {
        const float *a = R(f, n), *c = R(f, s);
        return ddy(a[0], c[0], a[1], a[-1], c[1], c[-1]);
    };

    typename L::template Copy<VEC, WALLS, PRE> copy;
    copy.init(T);
    // copy number j of the tile: gather row y0 - 3 + j, or record row y0 - 4 + j
    auto issue = [&](int j) {
        const int r = r_first + (L::kDecode ? 2 : 0) + j;
        if (j < rows + (L::kDecode ? 8 : 6) && row_ok(r)) copy.issue(T, pop_addr + static_cast<unsigned>(j % L::kSlots * L::kSlotBytes), r);
        cp_commit();
    };
#pragma unroll
    for (int j = 0; j < L::kSlots - 1; ++j) issue(j);

    // diagnostics: up to eight rows' sums, and the fastest node so far (the FP32 forms
    // spill 16 to 28 bytes for them)
    Sum3 sum_mass, sum_mom;
    Fastest fastest;
    // what the later stages of this column need.  f, rho_R, rho_B and j: before an
    // even iteration slots 0 .. 3 hold rows r - 1 .. r - 4, before an odd one
    // slots 1, 0, 3, 2; grad rho^N and G alternate
    float f[4][9], rr[4], rb[4], jx[4], jy[4], gx[2], gy[2], Gx[2], Gy[2];

    auto iteration = [&](auto C, const int k) {
        constexpr int c0 = decltype(C)::value;                    // ring slot of row r: k mod 2
        constexpr int old = 3 - c0, now = 1 - c0;                 // FIFO slots of rows r - 4 and r - 2, of row r
        constexpr int c1 = (c0 + 3) & 3, c2 = (c0 + 2) & 3, c3 = (c0 + 1) & 3;  // of rows r - 1, r - 2, r - 3
        const int r = r_first + k;
        if (!L::kDecode) cp_wait<L::kSlots - 2>();
        if constexpr (MODE == Pass::Fields) {  // read by D; its last readers are two barriers back
            density[t] = rr[old];
            density[W + t] = rb[old];
        }
        __syncthreads();
        issue(k + L::kSlots - 1);  // into the slot read in the last iteration
        // ---- D: row r - 4 (FIFO slot c0): rows r - 3, r - 4, r - 5 of the rings in slots c3, c0, c1
        const int yd = r - 4;
        if constexpr (MODE == Pass::Fields) {
            // thread t writes own column t (window column t + 4): warps then start on
            // 32-byte sectors, which host memory wants (page-locked outputs, 8192^2: 8.02
            // ms, 8.95 where each thread wrote its own column; device outputs the same)
            if (k >= 7 + kLead && t < W - 2 * kHalo && T.x0 + t < T.nx) {
                const size_t o = static_cast<size_t>(yd) * T.nx + (T.x0 + t);
                const float drr = density[t + kHalo], drb = density[W + t + kHalo];
                if (fo.rho_r) fo.rho_r[o] = drr;
                if (fo.rho_b) fo.rho_b[o] = drb;
                if (fo.ux) fo.ux[o] = R(kUx, c0)[kHalo];
                if (fo.uy) fo.uy[o] = R(kUy, c0)[kHalo];
                if (fo.p) fo.p[o] = fmaf(P.cs2_r, drr, P.cs2_b * drb);
            }
        } else if (k >= 7 + kLead && own_col) {
            const float drr = rr[old], drb = rb[old];
            const float rho = drr + drb;
            const float ux = R(kUx, c0)[0], uy = R(kUy, c0)[0];
            if (kStep) {
                if (!isfinite(rho)) atomicOr(T.flag, 1u);
                const float dPx = dx(kPhi, c3, c0, c1), dPy = dy(kPhi, c3, c1);
                const float divu = dx(kUx, c3, c0, c1) + dy(kUy, c3, c1);
                const float inv_rho = rcp(rho);
                const float nu = node_viscosity(drr, drb, inv_rho, P);
                float fp[9];
                collide_increment(f[old], drr, drb, rho, nu, ux, uy, Gx[c0], Gy[c0], dPx, dPy, divu, P, fp);
                const float ex = -R(kNx, c0)[0];
                const float ey = -R(kNy, c0)[0];
                const float phim = fmaf(P.kphi_r, drr, P.kphi_b * drb) * inv_rho;
                const float sg = P.beta * (drr * drb) * inv_rho * phim;
                if constexpr (L::kDecode)
                    L::Record::store(T.dst, T.nodes, static_cast<size_t>(yd) * T.nx, gx_own, fp, drr, drb, inv_rho, sg * ex,
                                     sg * ey, fmaf(0.5f * Gx[c0], inv_rho, ux), fmaf(0.5f * Gy[c0], inv_rho, uy), P);
                else
                    store_recoloured_f32(reinterpret_cast<float*>(T.dst) + static_cast<size_t>(yd) * T.nx, gx_own, T.nodes,
                                         fp, drr, drb, inv_rho, sg * ex, sg * ey);
            } else {
                const float* F = f[old];
                const float mx = (F[1] + F[7] + F[8]) - (F[3] + F[4] + F[5]);
                const float my = (F[1] + F[2] + F[3]) - (F[5] + F[6] + F[7]);
                if (isfinite(rho)) {
                    // (values whose FP32 sums or squares could overflow or underflow go to FP64)
                    if (fmaxf(fmaxf(fabsf(drr), fabsf(drb)), fmaxf(fabsf(mx), fabsf(my))) < 1e30f) {
                        sum_mass.add(drr, drb);
                        sum_mom.add(mx, my);
                    } else {
                        acc.r += drr;
                        acc.b += drb;
                        acc.jx += mx;
                        acc.jy += my;
                    }
                    fastest.add(ux, uy, acc.u2);
                } else {
                    acc.bad += 1.0;
                }
            }
        }
#pragma unroll
        for (int i = 0; i < 9; ++i) f[old][i] = f[now][i];  // row r - 2
        rr[old] = rr[now];
        rb[old] = rb[now];
        jx[old] = jx[now];
        jy[old] = jy[now];
        // ---- A: moments of row r
        if (k >= kLead && k <= rows + 5 + kLead && row_ok(r)) {
            const bool low = at_low(r), high = at_high(r);
            float fr[9], fb[9];
            // a link that comes from a wall is the node's own reversed link: an FP32
            // slot holds it in the link's place, decoded rows in its own
            auto gather = [&](auto edge) {
                constexpr bool kEdge = decltype(edge)::value;
#pragma unroll
                for (int i = 0; i < 9; ++i) {
                    const bool wall = kEdge && ((lcy(i) > 0 && low) || (lcy(i) < 0 && high));
                    const int d = PRE || wall ? 0 : -lcx(i);
                    if constexpr (L::kDecode) {
                        constexpr int s2 = c0 & 1;
                        // c1 = 3 - c0 of the four rows of c_y = 1: the later half
                        const int own = L::dec_row(lopp(i)) * W + (lcy(i) < 0 ? c0 * W + half : s2 * W);
                        const int row = L::dec_row(i) * W + (lcy(i) > 0 ? (c1 & 1) * W + ((c1 & 2) ? 2 * W - half : half)
                                                                        : (lcy(i) < 0 ? s2 ^ 1 : s2) * W);
                        const float2 v = dec[(wall ? own : row) + d];
                        fr[i] = v.x;
                        fb[i] = v.y;
                    } else {
                        const float* at = reinterpret_cast<const float*>(smem + k % L::kSlots * L::kSlotBytes) + t + d;
                        fr[i] = at[i * W];
                        fb[i] = at[(9 + i) * W];
                    }
                }
            };
            if (WALLS && !PRE && (low || high)) gather(std::true_type{});
            else gather(std::false_type{});
            const float2 rrb = sum9x2(fr, fb);
            const float arr = rrb.x, arb = rrb.y;
            const float ajx = ((fr[1] + fb[1]) + (fr[7] + fb[7])) + (fr[8] + fb[8]) -
                              (((fr[3] + fb[3]) + (fr[5] + fb[5])) + (fr[4] + fb[4]));
            const float ajy = ((fr[1] + fb[1]) + (fr[3] + fb[3])) + (fr[2] + fb[2]) -
                              (((fr[5] + fb[5]) + (fr[7] + fb[7])) + (fr[6] + fb[6]));
            const float a = arr * P.inv_rho0_r;
            const float b = arb * P.inv_rho0_b;
            const float inv_ab = rcp(__fadd_rn(a, b));
            const float chr = a * inv_ab;
            const float chb = b * inv_ab;
            R(kChiR, c0)[0] = chr;
            R(kChiB, c0)[0] = chb;
#pragma unroll
            for (int i = 0; i < 9; ++i) f[now][i] = fr[i] + fb[i];
            rr[now] = arr;
            rb[now] = arb;
            jx[now] = ajx;
            jy[now] = ajy;
            if (owned(k, 0)) {
                fwd(kFwdRR, r) = arr;
                fwd(kFwdRB, r) = arb;
                fwd(kFwdCHR, r) = chr;
                fwd(kFwdCHB, r) = chb;
            }
            if (at_low(r)) {
                R(kChiR, c1)[0] = chr;
                R(kChiB, c1)[0] = chb;
            }
            if (at_high(r)) {
                R(kChiR, c3)[0] = chr;
                R(kChiB, c3)[0] = chb;
            }
        }
        if (L::kDecode) cp_wait<L::kSlots - 1>();
        __syncthreads();
        // ---- E: record row r + 2, decoded (16-bit storage)
        if constexpr (L::kDecode) {
            const int ye = r + 2;
            if (k < rows + 8 && row_ok(ye))
                L::decode(smem + k % L::kSlots * L::kSlotBytes, t, dec, (c2 & 1) * W + 2 * W - half, (c0 & 1) * W, P);
        }
        // ---- B: row r - 1
        const int yb = r - 1;
        if (k >= 2 + kLead && k <= rows + 5 + kLead && row_ok(yb)) {
            const bool use_b = R(kChiR, c1)[0] > 0.5f;
            const int ch = use_b ? 4 * W : 0;
            const float *n_ = R(kChiR, c0) + ch, *m_ = R(kChiR, c1) + ch, *s_ = R(kChiR, c2) + ch;
            const float two = use_b ? -2.0f : 2.0f;
            const float bgx = two * ddx(m_[1], m_[-1], n_[1], n_[-1], s_[1], s_[-1]);
            const float bgy = two * ddy(n_[0], s_[0], n_[1], n_[-1], s_[1], s_[-1]);
            const float mag2 = fmaf(bgx, bgx, bgy * bgy);
            const float inv = (mag2 >= kNormalTau * kNormalTau) ? rsqrtf(mag2) : 0.0f;
            const float nhx = -bgx * inv;
            const float nhy = -bgy * inv;
            gx[c0] = bgx;
            gy[c0] = bgy;
            R(kNx, c1)[0] = nhx;
            R(kNy, c1)[0] = nhy;
            if (owned(k, 1)) {
                fwd(kFwdGX, yb) = bgx;
                fwd(kFwdGY, yb) = bgy;
            }
            if (at_low(yb)) {
                R(kNx, c2)[0] = nhx;
                R(kNy, c2)[0] = -nhy;
            }
            if (at_high(yb)) {
                R(kNx, c0)[0] = nhx;
                R(kNy, c0)[0] = -nhy;
            }
        }
        __syncthreads();
        // ---- C: row r - 2
        const int yc = r - 2;
        if (k >= 4 + kLead && k <= rows + 5 + kLead && row_ok(yc)) {
            const float K = P.curvature_mode == 0 ? dx(kNx, c1, c2, c3) + dy(kNy, c1, c3) : P.fixed_K;
            const float rho = rr[old] + rb[old];
            const float hk = P.half_sigma * K;
            const float cGx = fmaf(hk, gx[1 - c0], fmaf(rho, P.gacc_x, P.gvol_x));
            const float cGy = fmaf(hk, gy[1 - c0], fmaf(rho, P.gacc_y, P.gvol_y));
            const float inv_rho = rcp(rho);
            const float ux = fmaf(0.5f, cGx, jx[old]) * inv_rho;
            const float uy = fmaf(0.5f, cGy, jy[old]) * inv_rho;
            const float phip = fmaf(P.phip_r, rr[old], P.phip_b * rb[old]);
            Gx[c0] = cGx;
            Gy[c0] = cGy;
            R(kUx, c2)[0] = ux;
            R(kUy, c2)[0] = uy;
            R(kPhi, c2)[0] = phip;
            if (owned(k, 2)) {
                fwd(kFwdPHIP, yc) = phip;
                fwd(kFwdK, yc) = K;
                fwd(kFwdGFX, yc) = cGx;
                fwd(kFwdGFY, yc) = cGy;
                fwd(kFwdUX, yc) = ux;
                fwd(kFwdUY, yc) = uy;
            }
            if (at_low(yc)) {
                R(kUx, c3)[0] = -ux;
                R(kUy, c3)[0] = -uy;
                R(kPhi, c3)[0] = phip;
            }
            if (at_high(yc)) {
                R(kUx, c1)[0] = -ux;
                R(kUy, c1)[0] = -uy;
                R(kPhi, c1)[0] = phip;
            }
        }
    };
    for (int k = 0; k < iters; k += 2) {
        iteration(Const<0>{}, k);
        if (k + 1 < iters) iteration(Const<1>{}, k + 1);
        half = 2 * W - half;
        if (MODE == Pass::Diag && ((k & 6) == 6 || k + 2 >= iters)) {
            sum_mass.take(acc.r, acc.b);
            sum_mom.take(acc.jx, acc.jy);
        }
    }
    if (MODE == Pass::Diag) fastest.take(acc.u2);
    cp_wait<0>();
}

// The CTA's diagnostics: warp shuffles, then across the CTA's warps in shared memory (the rings are done).
template <int NT>
__device__ __forceinline__ void reduce_diag(const DiagAcc& acc, char* smem, double* __restrict__ partials) {
    const int t = threadIdx.x;
    double v[kDiagSlots] = {acc.r, acc.b, acc.jx, acc.jy, acc.u2, acc.bad};
#pragma unroll
    for (int j = 0; j < kDiagSlots; ++j) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            const double o = __shfl_down_sync(0xffffffffu, v[j], off);
            v[j] = (j == 4) ? fmax(v[j], o) : v[j] + o;
        }
    }
    __syncthreads();
    double* red = reinterpret_cast<double*>(smem);
    const int warp = t >> 5, lane = t & 31;
    if (lane == 0) {
#pragma unroll
        for (int j = 0; j < kDiagSlots; ++j) red[warp * kDiagSlots + j] = v[j];
    }
    __syncthreads();
    if (t < kDiagSlots) {
        double total = red[t];
        for (int w = 1; w < NT / 32; ++w) {
            const double o = red[w * kDiagSlots + t];
            total = (t == 4) ? fmax(total, o) : total + o;
        }
        partials[(static_cast<size_t>(blockIdx.y) * gridDim.x + blockIdx.x) * kDiagSlots + t] = total;
    }
}

template <class L, bool VEC, bool WALLS, Pass MODE, bool PRE>
__global__ void __launch_bounds__(L::W, march_ctas<L::W>())
    k_march(const char* __restrict__ src, char* __restrict__ dst, const StepParams P, const int rows, FieldOut fo,
            unsigned* __restrict__ flag, double* __restrict__ partials) {
    pdl_begin();
    extern __shared__ __align__(16) char smem[];
    DiagAcc acc;
    const int x0 = static_cast<int>(blockIdx.x) * (L::W - 2 * kHalo), y0 = static_cast<int>(blockIdx.y) * rows;
    const Tile T(src, dst, flag, P, x0, y0, rows);
    march_tile<L, VEC, WALLS, MODE, PRE>(smem, T, P, fo, acc);
    if (MODE == Pass::Diag) reduce_diag<L::W>(acc, smem, partials);
}

// ---------------------------------------------------------------------------
// Small lattices, FP32 storage: one node per thread, no marching.
//
// A lattice that does not fill the GPU is bound by latency: the march takes
// rows + 7 iterations of about 0.75 us, however few its rows.  Here a CTA
// takes a window of 32 x H nodes (26 x (H - 6) of them its own), each thread
// gathers its node straight from L2 into registers and runs all four stages
// of it, with three barriers and no copies in between, so that a step is one
// load latency, four short stages and the launch.  The window's halo costs
// 2x (H = 16) to 5x (H = 8) the arithmetic and L2 reads, which idle SMs have
// to spare.  The arithmetic is the march's, expression by expression: both
// give the same bits.
// Measured per step, march -> this kernel: 64^2 6.5 -> 2.05 us, 128^2 7.7 -> 2.75,
// 256^2 10.3 -> 4.2, 1024 x 128 10.9 -> 7.2, 512^2 21 -> 12.4.
//
// 16-bit storage: each thread first decodes its node's record into FP32
// populations in shared memory (one more halo node and barrier: 24 x (H - 8)
// own nodes), and stage A gathers from there.
// ---------------------------------------------------------------------------
constexpr int kSmallX = 32;  // window columns: one warp per window row
template <class L>
constexpr int small_halo() { return L::kDecode ? 4 : 3; }
// fields of the window in shared memory: chi_R, chi_B, Phi', n-hat x, y, u x, y;
// with 16-bit storage the last four take the place of decoded populations, which
// only stage A reads
template <class L>
constexpr int small_fields() { return L::kDecode ? 3 + kPlanes : 7; }

template <class L, int H, bool WALLS, Pass MODE>
__global__ void __launch_bounds__(kSmallX * H, 1024 / (kSmallX * H))
    k_small(const char* __restrict__ state, char* __restrict__ dst, const StepParams P, FieldOut fo,
            unsigned* __restrict__ flag) {
    pdl_begin();
    constexpr int kN = kSmallX * H;
    constexpr int kEdge = small_halo<L>();
    __shared__ float sm[small_fields<L>() * kN + 2 * kSmallX];
    const int tx = threadIdx.x % kSmallX, ty = threadIdx.x / kSmallX;
    const int nx = P.nx, ny = P.ny;
    const size_t nodes = static_cast<size_t>(nx) * ny;
    // this thread's node (its periodic image in the lattice)
    const int xw = static_cast<int>(blockIdx.x) * (kSmallX - 2 * kEdge) - kEdge + tx;
    const int yw = static_cast<int>(blockIdx.y) * (H - 2 * kEdge) - kEdge + ty;
    const int x = wrap(xw, nx), y = WALLS ? yw : wrap(yw, ny);
    const bool in = !WALLS || (y >= 0 && y < ny);
    const bool low = WALLS && y == 0, high = WALLS && y == ny - 1;
    float* w = sm + kSmallX + threadIdx.x;  // this node in a field of the window
    constexpr int kChiR = 0, kChiB = 1, kPhi = 2, kNx = 3, kNy = 4, kUx = 5, kUy = 6;
    // rows above and below in the window; beyond a wall the node's own row, odd fields negated
    const int up = high ? 0 : kSmallX, dn = low ? 0 : -kSmallX;
    auto dx = [&](const float* a, float pu, float pd) {
        return ddx(a[1], a[-1], WALLS ? pu * a[up + 1] : a[up + 1], WALLS ? pu * a[up - 1] : a[up - 1],
                   WALLS ? pd * a[dn + 1] : a[dn + 1], WALLS ? pd * a[dn - 1] : a[dn - 1]);
    };
    auto dy = [&](const float* a, float pu, float pd) {
        return ddy(WALLS ? pu * a[up] : a[up], WALLS ? pd * a[dn] : a[dn], WALLS ? pu * a[up + 1] : a[up + 1],
                   WALLS ? pu * a[up - 1] : a[up - 1], WALLS ? pd * a[dn + 1] : a[dn + 1],
                   WALLS ? pd * a[dn - 1] : a[dn - 1]);
    };
    const float ou = high ? -1.0f : 1.0f, od = low ? -1.0f : 1.0f;  // parity of odd fields

    float* pop = w + 3 * kN;  // this node's decoded populations (16-bit storage)
    if constexpr (L::kDecode) {
        if (in) {
            float2 v[9];
            L::Record::load(state, nodes, static_cast<size_t>(y) * nx, x, P, v);
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                pop[i * kN] = v[i].x;
                pop[(9 + i) * kN] = v[i].y;
            }
        }
        __syncthreads();
    }
    // ---- A
    float f[9], rr = 1.0f, rb = 1.0f, jx = 0.0f, jy = 0.0f, chr = 0.0f, chb = 0.0f;
    const bool in_a = in && (!L::kDecode || (tx >= 1 && tx < kSmallX - 1 && ty >= 1 && ty < H - 1));
    if (in_a) {
        float fr[9], fb[9];
        if constexpr (L::kDecode) {
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                const bool wall = WALLS && ((lcy(i) > 0 && low) || (lcy(i) < 0 && high));
                const float* at = pop + (wall ? lopp(i) * kN : i * kN - lcy(i) * kSmallX - lcx(i));
                fr[i] = at[0];
                fb[i] = at[9 * kN];
            }
        } else {
            const float* src = reinterpret_cast<const float*>(state);
            const unsigned xm = x == 0 ? nx - 1 : x - 1, xp = x == nx - 1 ? 0 : x + 1;
            const unsigned ym = y == 0 ? ny - 1 : y - 1, yp = y == ny - 1 ? 0 : y + 1;
            const unsigned o = static_cast<unsigned>(y) * nx + x;
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                unsigned at = (lcy(i) > 0 ? ym : (lcy(i) < 0 ? yp : static_cast<unsigned>(y))) * nx +
                              (lcx(i) > 0 ? xm : (lcx(i) < 0 ? xp : static_cast<unsigned>(x)));
                int li = i;
                if (WALLS && ((lcy(i) > 0 && low) || (lcy(i) < 0 && high))) {
                    li = lopp(i);
                    at = o;
                }
                fr[i] = __ldcg(src + nodes * li + at);
                fb[i] = __ldcg(src + nodes * (9 + li) + at);
            }
        }
        const float2 rrb = sum9x2(fr, fb);
        rr = rrb.x;
        rb = rrb.y;
        jx = ((fr[1] + fb[1]) + (fr[7] + fb[7])) + (fr[8] + fb[8]) -
             (((fr[3] + fb[3]) + (fr[5] + fb[5])) + (fr[4] + fb[4]));
        jy = ((fr[1] + fb[1]) + (fr[3] + fb[3])) + (fr[2] + fb[2]) -
             (((fr[5] + fb[5]) + (fr[7] + fb[7])) + (fr[6] + fb[6]));
        const float a = rr * P.inv_rho0_r;
        const float b = rb * P.inv_rho0_b;
        const float inv_ab = rcp(__fadd_rn(a, b));
        chr = a * inv_ab;
        chb = b * inv_ab;
        w[kChiR * kN] = chr;
        w[kChiB * kN] = chb;
#pragma unroll
        for (int i = 0; i < 9; ++i) f[i] = fr[i] + fb[i];
    }
    const float phip = fmaf(P.phip_r, rr, P.phip_b * rb);
    w[kPhi * kN] = phip;
    __syncthreads();
    // ---- B
    float gx = 0.0f, gy = 0.0f, nhx = 0.0f, nhy = 0.0f;
    constexpr int kB = kEdge - 2, kC = kEdge - 1;
    const bool in_b = in && tx >= kB && tx < kSmallX - kB && ty >= kB && ty < H - kB;
    if (in_b) {
        const bool use_b = chr > 0.5f;
        const float* ch = w + (use_b ? kChiB * kN : 0);
        const float two = use_b ? -2.0f : 2.0f;
        gx = two * dx(ch, 1.0f, 1.0f);
        gy = two * dy(ch, 1.0f, 1.0f);
        const float mag2 = fmaf(gx, gx, gy * gy);
        const float inv = (mag2 >= kNormalTau * kNormalTau) ? rsqrtf(mag2) : 0.0f;
        nhx = -gx * inv;
        nhy = -gy * inv;
        w[kNx * kN] = nhx;
        w[kNy * kN] = nhy;
    }
    __syncthreads();
    // ---- C
    float K = 0.0f, Gx = 0.0f, Gy = 0.0f, ux = 0.0f, uy = 0.0f;
    const bool in_c = in && tx >= kC && tx < kSmallX - kC && ty >= kC && ty < H - kC;
    if (in_c) {
        K = P.curvature_mode == 0 ? dx(w + kNx * kN, 1.0f, 1.0f) + dy(w + kNy * kN, ou, od) : P.fixed_K;
        const float rho = rr + rb;
        const float hk = P.half_sigma * K;
        Gx = fmaf(hk, gx, fmaf(rho, P.gacc_x, P.gvol_x));
        Gy = fmaf(hk, gy, fmaf(rho, P.gacc_y, P.gvol_y));
        const float inv_rho = rcp(rho);
        ux = fmaf(0.5f, Gx, jx) * inv_rho;
        uy = fmaf(0.5f, Gy, jy) * inv_rho;
        w[kUx * kN] = ux;
        w[kUy * kN] = uy;
    }
    __syncthreads();
    // ---- D
    if (!(in && tx >= kEdge && tx < kSmallX - kEdge && ty >= kEdge && ty < H - kEdge && xw < nx && yw < ny)) return;
    const size_t row = static_cast<size_t>(y) * nx;
    if (MODE == Pass::StepFields || MODE == Pass::FwdFields) {
        float* o = fo.fwd + row + x;
        o[kFwdRR * nodes] = rr;
        o[kFwdRB * nodes] = rb;
        o[kFwdCHR * nodes] = chr;
        o[kFwdCHB * nodes] = chb;
        o[kFwdPHIP * nodes] = phip;
        o[kFwdGX * nodes] = gx;
        o[kFwdGY * nodes] = gy;
        o[kFwdK * nodes] = K;
        o[kFwdGFX * nodes] = Gx;
        o[kFwdGFY * nodes] = Gy;
        o[kFwdUX * nodes] = ux;
        o[kFwdUY * nodes] = uy;
        if (MODE == Pass::FwdFields) return;
    }
    const float rho = rr + rb;
    if (!isfinite(rho)) atomicOr(flag, 1u);
    const float dPx = dx(w + kPhi * kN, 1.0f, 1.0f), dPy = dy(w + kPhi * kN, 1.0f, 1.0f);
    const float divu = dx(w + kUx * kN, ou, od) + dy(w + kUy * kN, ou, od);
    const float inv_rho = rcp(rho);
    const float nu = node_viscosity(rr, rb, inv_rho, P);
    float fp[9];
    collide_increment(f, rr, rb, rho, nu, ux, uy, Gx, Gy, dPx, dPy, divu, P, fp);
    const float ex = -nhx, ey = -nhy;
    const float phim = fmaf(P.kphi_r, rr, P.kphi_b * rb) * inv_rho;
    const float sg = P.beta * (rr * rb) * inv_rho * phim;
    if constexpr (L::kDecode)
        L::Record::store(dst, nodes, row, x, fp, rr, rb, inv_rho, sg * ex, sg * ey, fmaf(0.5f * Gx, inv_rho, ux),
                         fmaf(0.5f * Gy, inv_rho, uy), P);
    else
        store_recoloured_f32(reinterpret_cast<float*>(dst) + row, x, nodes, fp, rr, rb, inv_rho, sg * ex, sg * ey);
}

template <class L, bool VEC, bool WALLS, Pass MODE, bool PRE>
cudaError_t launch_march_one(const void* src, void* dst, const StepParams& P, int rows, FieldOut fo, unsigned* flag,
                             double* partials, cudaStream_t s) {
    static std::atomic<unsigned long long> configured{0};  // per device, set from any host thread
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = 1ull << (dev & 63);
    if (!(configured.load() & bit)) {
        e = cudaFuncSetAttribute(k_march<L, VEC, WALLS, MODE, PRE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 L::kBytes);
        if (e != cudaSuccess) return e;
        configured.fetch_or(bit);
    }
    return launch_pdl(k_march<L, VEC, WALLS, MODE, PRE>, chain_grid(P.nx, P.ny, rows), dim3(L::W), L::kBytes, s,
                      static_cast<const char*>(src), static_cast<char*>(dst), P, rows, fo, flag, partials);
}

template <class L>
dim3 small_grid(const StepParams& P, int H) {
    const int tx = kSmallX - 2 * small_halo<L>(), ty = H - 2 * small_halo<L>();
    return dim3(static_cast<unsigned>((P.nx + tx - 1) / tx), static_cast<unsigned>((P.ny + ty - 1) / ty));
}

// Whether a step runs as k_small: up to where the march, whose copies are of 4
// bytes where nx is no multiple of 4, becomes the faster on average.  Per step,
// k_small against the march:
//   FP32, 16-byte copies: 640^2 18.3 and 19.4 us, 700^2 21.4 and 20.5, 1024 x 512
//     22.8 and 23.0, 256 x 2048 22.6 and 25.5, 736^2 24.1 and 22.2, 776 x 772 26.9
//     and 21.9;
//   FP32, 4-byte: 653^2 19.4 and 20.9, 721^2 22.7 and 24.2, 763^2 26.0 and 25.6, 491
//     x 1201 26.1 and 27.6, 775^2 27.0 and 26.4, 801^2 29.8 and 26.5, 837^2 34.0 and 28.6;
//   FP16, 16-byte: 512^2 16.7 and 17.8, 540^2 18.5 and 17.7, 1024 x 300 18.6 and
//     19.3, 576^2 19.7 and 19.1, 640^2 24.3 and 23.1;
//   FP16, 4-byte: 575^2 20.4 and 21.7, 601^2 23.0 and 26.1, 655^2 26.6 and 27.3.
template <class L>
bool use_small(const StepParams& P) {
    const bool vec = (P.nx % 4) == 0;
    const long limit = L::kDecode ? (vec ? 330000 : 430000) : (vec ? 530000 : 600000);
    const int rows = 16 - 2 * small_halo<L>();
    return static_cast<long>(P.nx) * P.ny <= limit && P.ny <= 65535 * rows;  // grid rows
}

// Window rows of k_small: a step takes about 1.7 us plus c ceil(tiles / SMs),
// c growing with the threads of a CTA (fits to 64^2 .. 512^2).
template <class L>
int small_rows(const StepParams& P) {
    struct Fit {
        int rows;
        double c;
    };
    constexpr Fit fits[3] = {{8, L::kDecode ? 1e30 : 0.45}, {10, L::kDecode ? 0.6 : 0.57}, {16, L::kDecode ? 1.3 : 1.2}};
    const long sms = 152;
    int best = 16;
    double best_cost = 1e30;
    for (const Fit& f : fits) {
        if (f.rows <= 2 * small_halo<L>()) continue;  // no rows of its own
        const dim3 g = small_grid<L>(P, f.rows);
        const double cost = f.c * ((static_cast<long>(g.x) * g.y + sms - 1) / sms);
        if (cost < best_cost && g.y <= 65535) {
            best_cost = cost;
            best = f.rows;
        }
    }
    return best;
}

template <class L, int H, Pass MODE>
cudaError_t launch_small(const void* src, void* dst, const StepParams& P, FieldOut fo, unsigned* flag,
                         cudaStream_t s) {
    const dim3 g = small_grid<L>(P, H);
    const char* a = static_cast<const char*>(src);
    char* b = static_cast<char*>(dst);
    if (P.wall_y) return launch_pdl(k_small<L, H, true, MODE>, g, dim3(kSmallX * H), 0, s, a, b, P, fo, flag);
    return launch_pdl(k_small<L, H, false, MODE>, g, dim3(kSmallX * H), 0, s, a, b, P, fo, flag);
}

template <class L, Pass MODE>
cudaError_t launch_small_any(const void* src, void* dst, const StepParams& P, FieldOut fo, unsigned* flag,
                             cudaStream_t s) {
    switch (small_rows<L>(P)) {
        case 8:
            if constexpr (!L::kDecode) return launch_small<L, 8, MODE>(src, dst, P, fo, flag, s);
            [[fallthrough]];
        case 10: return launch_small<L, 10, MODE>(src, dst, P, fo, flag, s);
        default: return launch_small<L, 16, MODE>(src, dst, P, fo, flag, s);
    }
}

template <class L, Pass MODE, bool PRE = false>
cudaError_t launch_march(const void* src, void* dst, const StepParams& P, int rows, FieldOut fo, unsigned* flag,
                         double* partials, cudaStream_t s) {
    if constexpr (MODE == Pass::Step || MODE == Pass::StepFields) {
        if (use_small<L>(P)) return launch_small_any<L, MODE>(src, dst, P, fo, flag, s);
    }
    const bool vec = (P.nx % 4) == 0;
    // 16-bit rows copied 4 bytes at a time take the form for walls, which is right for
    // any lattice: the periodic one spills 12 bytes, and its copies through L1 evict
    // them (BF16 3883 x 634 180 us per step against 116)
    const bool walls = P.wall_y != 0 || (L::kDecode && !vec);
    if (vec && walls) return launch_march_one<L, true, true, MODE, PRE>(src, dst, P, rows, fo, flag, partials, s);
    if (vec) return launch_march_one<L, true, false, MODE, PRE>(src, dst, P, rows, fo, flag, partials, s);
    if constexpr (!L::kDecode) {
        if (!walls) return launch_march_one<L, false, false, MODE, PRE>(src, dst, P, rows, fo, flag, partials, s);
    }
    return launch_march_one<L, false, true, MODE, PRE>(src, dst, P, rows, fo, flag, partials, s);
}

}  // namespace
}  // namespace cmrt
