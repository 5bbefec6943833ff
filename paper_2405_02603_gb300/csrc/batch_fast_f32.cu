// batch_fast_f32.cu -- the persistent batched kernel on the specialised FP32
// passes (fast.cuh): the scheme of batch.cu (pass-major work list, an atomic
// cursor, bounded waits on the previous pass's count), each tile by its
// size's register-resident body instead of the generic engine.
//
// Every body runs in 128 threads, so that one CTA shape serves all sizes and
// passes: a tile has 128 / (n / V) lines.  Four CTAs per SM: 64 solves of mixed
// N in 3.02 ms; with three (168 registers, nothing spilled) 3.42, with five
// (96) 3.45, with six 3.92; the generic engine's kernel takes 9.07.  A work
// item is a run of tiles of one pass of about 8K points: the cursor, the item's
// descriptor and the wait are paid for once per item.
#include <algorithm>
#include <cuda/atomic>

#include "../../include/fsp.h"
#include "batch_fast.h"
#include "fast.cuh"

namespace fsp {
namespace fast {
namespace {

constexpr int kThreads = 128;
constexpr int kItemPoints = 8192;

template <int N> struct BRow {
    using K = Cfg<float, N>;
    static constexpr int V = K::V, L = kThreads / (N / K::V), R1 = K::R1, R2 = K::R2, R3 = K::R3;
    static constexpr bool lane = LaneRow<float, N, V, R1, R2, R3>::ok;
    static constexpr int tiles = (N * N + L - 1) / L;
    static constexpr int group = kItemPoints / (L * N) > 1 ? kItemPoints / (L * N) : 1;
    static constexpr size_t smem() {
        if constexpr (lane)
            return lane_row_smem<float, N, V, L>();
        else
            return (size_t)(N + 1) * (L + 1) * sizeof(float2);
    }
};
// lines of 96: 12 values per thread, since 16 lines of 24 would leave half of
// the 128 threads out and 32 lines do not divide 48
template <int n> struct BColCfg : Cfg<float, n> {};
template <> struct BColCfg<96> {
    static constexpr int V = 12, R1 = 4, R2 = 6, R3 = 4;
};
template <int N> struct BCol {
    static constexpr int n = 2 * N;
    using K = BColCfg<n>;
    static constexpr int V = K::V, L = kThreads / (n / V), R1 = K::R1, R2 = K::R2, R3 = K::R3;
    static_assert(N % L == 0, "tiles must cover k_x < N exactly");
    static constexpr int tiles = N / L * (N + 1);  // P2, P4; twice as many in P3
    static constexpr int group = kItemPoints / (L * n) > 1 ? kItemPoints / (L * n) : 1;
    static constexpr size_t smem() {
        return sizeof(float2) * n * (L + 1) + (ColOpt<float, COL_FMI, n>::TWS ? sizeof(float2) * n : 0);
    }
};

template <int N> __device__ __noinline__ void row_r2c(const RowArgs &a, int tile) {
    using B = BRow<N>;
    if constexpr (B::lane)
        lane_r2c_tile<float, N, B::V, B::L, B::R1>(a, tile);
    else
        fast_r2c_tile<float, N, B::V, B::L, B::R1, B::R2, B::R3>(a, tile);
}
template <int N> __device__ __noinline__ void row_c2r(const RowArgs &a, int tile) {
    using B = BRow<N>;
    if constexpr (B::lane)
        lane_c2r_tile<float, N, B::V, B::L, B::R1, true>(a, tile);
    else
        fast_c2r_tile<float, N, B::V, B::L, B::R1, B::R2, B::R3, true>(a, tile);
}
template <int N, int MODE> __device__ __noinline__ void col(const ColArgs &a, int tile) {
    using B = BCol<N>;
    fast_col_body<float, B::n, B::V, B::L, B::R1, B::R2, B::R3, MODE, false>(a, tile % (N / B::L), tile / (N / B::L));
}

template <int N> __device__ __forceinline__ void solve_tile(int pass, const RowArgs &r, const ColArgs &c, int tile) {
    switch (pass) {
    case 0: row_r2c<N>(r, tile); break;
    case 1: col<N, COL_FWD>(c, tile); break;
    case 2: col<N, COL_FMI>(c, tile); break;
    case 3: col<N, COL_INV>(c, tile); break;
    default: row_c2r<N>(r, tile); break;
    }
}

__device__ __forceinline__ unsigned long long batch_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__global__ void __launch_bounds__(kThreads, 4) k_batch_fast(const FastBatchLaunch L) {
    __shared__ int s_stop, s_n, s_pass, s_first, s_last, s_done;
    __shared__ __align__(16) RowArgs s_row;
    __shared__ __align__(16) ColArgs s_col;
    for (;;) {
        if (threadIdx.x == 0) {
            cuda::atomic_ref<int, cuda::thread_scope_device> status(L.ctl->status);
            int stop = 1;
            if (status.load(cuda::memory_order_relaxed) == 0) {
                const int item = atomicAdd(&L.ctl->cursor, 1);
                if (item < L.total) {
                    stop = 0;
                    const FastBatchItem it = L.items[item];
                    const BatchSeg g = L.segs[it.seg];
                    const FastBatchSolve &sv = L.solves[g.solve];
                    s_n = sv.N, s_pass = g.pass, s_done = g.solve * 5 + g.pass;
                    // g.ntiles holds the segment's tiles; an item ends where the next one begins
                    s_first = it.tile0;
                    s_last = item + 1 < L.total && L.items[item + 1].seg == it.seg ? L.items[item + 1].tile0 : g.ntiles;
                    if (g.pass == 0 || g.pass == 4)
                        s_row = g.pass == 0 ? sv.r1 : sv.r5;
                    else
                        s_col = g.pass == 1 ? sv.c2 : g.pass == 2 ? sv.c3 : sv.c4;
                    if (g.pass > 0) {
                        cuda::atomic_ref<int, cuda::thread_scope_device> prev(L.ctl->done[g.solve * 5 + g.pass - 1]);
                        const unsigned long long t0 = batch_ns();
                        unsigned sleep = 32;
                        while (prev.load(cuda::memory_order_acquire) < g.need_prev) {
                            if (status.load(cuda::memory_order_relaxed) != 0) {
                                stop = 1;
                                break;
                            }
                            if (batch_ns() - t0 > L.timeout_ns) {
                                int expected = 0;
                                status.compare_exchange_strong(expected, (int)FSP_ETIMEOUT);
                                stop = 1;
                                break;
                            }
                            __nanosleep(sleep);
                            if (sleep < 2048) sleep <<= 1;
                        }
                    }
                }
            }
            s_stop = stop;
        }
        __syncthreads();
        if (s_stop) break;
        const int n = s_n, pass = s_pass, last = s_last;
        for (int tile = s_first; tile < last; ++tile) {
            switch (n) {
            case 32: solve_tile<32>(pass, s_row, s_col, tile); break;
            case 48: solve_tile<48>(pass, s_row, s_col, tile); break;
            case 64: solve_tile<64>(pass, s_row, s_col, tile); break;
            case 96: solve_tile<96>(pass, s_row, s_col, tile); break;
            case 128: solve_tile<128>(pass, s_row, s_col, tile); break;
            case 160: solve_tile<160>(pass, s_row, s_col, tile); break;
            case 192: solve_tile<192>(pass, s_row, s_col, tile); break;
            default: solve_tile<256>(pass, s_row, s_col, tile); break;
            }
            __syncthreads();  // the tile's shared memory is free, its stores are ordered before the count
        }
        if (threadIdx.x == 0) {
            __threadfence();
            cuda::atomic_ref<int, cuda::thread_scope_device> d(L.ctl->done[s_done]);
            d.fetch_add(1, cuda::memory_order_release);
        }
    }
}

template <int N> void tiles_of(int ntiles[5], int group[5]) {
    using R = BRow<N>;
    using C = BCol<N>;
    ntiles[0] = ntiles[4] = R::tiles, group[0] = group[4] = R::group;
    ntiles[1] = ntiles[3] = C::tiles, group[1] = group[3] = C::group;
    ntiles[2] = 2 * C::tiles, group[2] = C::group > 1 ? C::group / 2 : 1;
}
template <int N> size_t smem_of() { return BRow<N>::smem() > BCol<N>::smem() ? BRow<N>::smem() : BCol<N>::smem(); }

}  // namespace
}  // namespace fast

bool fast_batch_has(int N) {
    return N == 32 || N == 48 || N == 64 || N == 96 || N == 128 || N == 160 || N == 192 || N == 256;
}
void fast_batch_tiles(int N, int ntiles[5], int group[5]) {
    switch (N) {
    case 32: fast::tiles_of<32>(ntiles, group); break;
    case 48: fast::tiles_of<48>(ntiles, group); break;
    case 64: fast::tiles_of<64>(ntiles, group); break;
    case 96: fast::tiles_of<96>(ntiles, group); break;
    case 128: fast::tiles_of<128>(ntiles, group); break;
    case 160: fast::tiles_of<160>(ntiles, group); break;
    case 192: fast::tiles_of<192>(ntiles, group); break;
    case 256: fast::tiles_of<256>(ntiles, group); break;
    }
}
size_t fast_batch_smem(int N) {
    switch (N) {
    case 32: return fast::smem_of<32>();
    case 48: return fast::smem_of<48>();
    case 64: return fast::smem_of<64>();
    case 96: return fast::smem_of<96>();
    case 128: return fast::smem_of<128>();
    case 160: return fast::smem_of<160>();
    case 192: return fast::smem_of<192>();
    case 256: return fast::smem_of<256>();
    }
    return 0;
}
// Sets the shared-memory attribute too, so that the launch can be captured: to
// what the largest size needs whatever this batch holds, because it is one
// value for the process and other live batches are captured again under it.
int fast_batch_blocks_per_sm(size_t smem) {
    int nb = 0;
    size_t most = 0;
    for (int N : {32, 48, 64, 96, 128, 160, 192, 256}) most = std::max(most, fast_batch_smem(N));
    cudaFuncSetAttribute(fast::k_batch_fast, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, fast::k_batch_fast, fast::kThreads, smem) != cudaSuccess)
        return 0;
    return nb;
}
cudaError_t launch_fast_batch(const FastBatchLaunch &L, cudaStream_t s) {
    fast::k_batch_fast<<<L.grid, fast::kThreads, L.smem, s>>>(L);
    return cudaGetLastError();
}

}  // namespace fsp
