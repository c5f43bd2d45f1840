// Batched ensembles: one persistent launch steps many lattices (the march of
// cmrt_march.cuh over a work list).
#include "cmrt_march.cuh"

namespace cmrt {
namespace {

// A persistent kernel over a work list of tiles of many independent lattices.
// Each CTA takes the next item (member, strip, row segment) from a global
// counter until the list is exhausted; every item is the row pipeline of
// k_march, with that member's own parameters and buffers, which it keeps in
// shared memory: held per thread they are some 60 registers more than the
// march has.  No CTA waits on another: an atomicAdd hands out the items, and the
// last CTA to leave resets the counters for the next launch.
//
// A strip's window is 96 or 128 columns wide (five or four CTAs per SM),
// whichever computes fewer columns over the batch: with sides of 64 to 512, 96
// cuts 512 into 6 x 88 and 256 into 3 x 88 own columns.  Measured, 512 periodic
// members of 64^2 .. 512^2, 64 rows per item: 1517 us per step before (the
// warp-specialised pipeline), 1233 us with 128 columns, 1150 us with 96; tuned
// rows 1416 -> 1096 us; FP16 1998 -> 1497 us.  WALLS (a batch with a walled
// member) runs one form of the pipeline for all members: with both forms in one
// kernel the compiler merges their common parts and spills (1898 us).
template <class L, bool VEC, bool WALLS>
__global__ void __launch_bounds__(L::W, 512 / L::W) k_batch(const BatchArgs A) {
    extern __shared__ __align__(16) char smem[];
    __shared__ __align__(16) StepParams P;
    __shared__ __align__(16) Tile T;
    __shared__ int s_item;
    const int t = threadIdx.x;
    for (;;) {
        __syncthreads();  // the previous item is done with the rings, P, T and s_item
        if (t == 0) s_item = static_cast<int>(atomicAdd(&A.counters[0], 1u));
        __syncthreads();
        const int it = s_item;
        if (it >= A.nitems) break;
        const BatchItem w = A.items[it];
        static_assert(sizeof(StepParams) / 4 <= 64, "one word per thread");
        if (t < static_cast<int>(sizeof(StepParams) / 4))
            reinterpret_cast<unsigned*>(&P)[t] = reinterpret_cast<const unsigned*>(A.params + w.member)[t];
        if (t == 64) {
            const StepParams& q = A.params[w.member];
            const size_t off = A.offsets[w.member];
            T = Tile(A.src + off, A.dst + off, A.flags + w.member, q, w.x0, w.y0, w.rows);
        }
        __syncthreads();
        DiagAcc acc;
        march_tile<L, VEC, WALLS, Pass::Step, false>(smem, T, P, FieldOut{}, acc);
    }
    if (t == 0) {
        __threadfence();  // this CTA's last counter access precedes its exit count
        const unsigned done = atomicAdd(&A.counters[1], 1u);
        if (done == gridDim.x - 1) {
            A.counters[0] = 0u;
            A.counters[1] = 0u;
            __threadfence();
        }
    }
}

template <class L, bool VEC, bool WALLS>
cudaError_t batch_configure(int dev, int* ctas_per_sm) {
    static std::atomic<unsigned long long> configured{0};  // per device, set from any host thread
    const unsigned long long bit = 1ull << (dev & 63);
    cudaError_t e = cudaSuccess;
    if (!(configured.load() & bit)) {
        e = cudaFuncSetAttribute(k_batch<L, VEC, WALLS>, cudaFuncAttributeMaxDynamicSharedMemorySize, L::kBytes);
        if (e != cudaSuccess) return e;
        configured.fetch_or(bit);
    }
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(ctas_per_sm, k_batch<L, VEC, WALLS>, L::W, L::kBytes);
}

template <class L, bool VEC, bool WALLS>
cudaError_t batch_launch(const BatchArgs& A, int grid, cudaStream_t s) {
    k_batch<L, VEC, WALLS><<<grid, L::W, L::kBytes, s>>>(A);
    return cudaGetLastError();
}

// f(layout, vec, walls) with the march's layout for a batch's form.  (16-bit rows copied
// 4 bytes at a time keep the periodic form here: without the tile in registers it does
// not spill, as it does in the kernel of one lattice; FP32 with walls spills 4 bytes.)
template <class F>
cudaError_t with_layout(const BatchForm& b, F&& f) {
    using Yes = std::true_type;
    using No = std::false_type;
    auto wide = [&](auto w) {
        constexpr int W = decltype(w)::value;
        auto go = [&](auto l) {
            if (b.walls) return b.vec ? f(l, Yes{}, Yes{}) : f(l, No{}, Yes{});
            return b.vec ? f(l, Yes{}, No{}) : f(l, No{}, No{});
        };
        switch (b.precision) {
            case kPrecF16: return go(March16<__half2, W>{});
            case kPrecB16: return go(March16<__nv_bfloat162, W>{});
            default: return go(MarchF32<W>{});
        }
    };
    return b.window == 96 ? wide(Const<96>{}) : wide(Const<kWin>{});
}

}  // namespace

cudaError_t prepare_batch(const BatchForm& b, int* ctas_per_sm) {
    int dev = 0;
    const cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    return with_layout(b, [&](auto l, auto v, auto w) {
        return batch_configure<decltype(l), decltype(v)::value, decltype(w)::value>(dev, ctas_per_sm);
    });
}

cudaError_t launch_batch(const BatchArgs& A, const BatchForm& b, int grid, cudaStream_t s) {
    return with_layout(b, [&](auto l, auto v, auto w) {
        return batch_launch<decltype(l), decltype(v)::value, decltype(w)::value>(A, grid, s);
    });
}

}  // namespace cmrt
