// Kernels of the row-partitioned FP64 SpMV (Sec. III-A, Fig. 3 of Pearson,
// Javeed and Devine): the Pack gather, the halo exchange copy, and the CSR
// products y_L = A_L x_L and y += A_R x_R.
//
// Design for sm_103a: FP64 FMA issues at 2 lanes/clk/SM on this part, so a
// CSR product with HBM at full speed is nearly FP64-bound.  The staged kernel
// therefore spends one DFMA per stored entry where a lane walks a row (in one or
// two sums), and gets coalescing from bulk copies (cp.async.bulk, the TMA
// engine) of whole tiles into a stage of shared memory per warp instead of from
// lanes cooperating on a row, which costs FP64 adds in shuffle reductions; long
// rows, where that costs little, go to a whole warp or a whole CTA.  Every row is
// summed in an order that depends on the matrix and the variant alone, so results
// do not depend on the grid, the stream or the schedule.
#include "internal.h"
#include "pdl.cuh"

#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>

namespace spmvk {

// ------------------------------------------------------------------------
// PTX helpers: mbarrier, bulk copy, global timer
// ------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ uint64_t global_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_fence_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t tx) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(tx)
                 : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
// Wait for phase `parity` of an mbarrier, giving up after limit_ns.
__device__ __forceinline__ bool mbar_wait_bounded(uint32_t bar, uint32_t parity,
                                                  uint64_t limit_ns) {
    if (mbar_try_wait(bar, parity)) return true;
    const uint64_t t0 = global_ns();
    while (!mbar_try_wait(bar, parity)) {
        if (global_ns() - t0 > limit_ns) return false;
    }
    return true;
}
// Bulk copy global -> shared (16-byte aligned addresses, size % 16 == 0) with an
// L2 eviction policy (evict-first for data read once), completion reported to
// an mbarrier as transaction bytes.
__device__ __forceinline__ void bulk_g2s_hint(uint32_t dst, const void* src, uint32_t bytes,
                                              uint32_t bar, uint64_t policy) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint "
        "[%0], [%1], %2, [%3], %4;" ::"r"(dst),
        "l"(src), "r"(bytes), "r"(bar), "l"(policy)
        : "memory");
}
__device__ __forceinline__ uint64_t policy_evict_first() {
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    return p;
}
__device__ __forceinline__ uint64_t policy_evict_last() {
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
    return p;
}
// Read-only load of x kept in L2 (x is gathered many times per product).
__device__ __forceinline__ double ldg_keep(const double* p, uint64_t policy) {
    double v;
    asm("ld.global.nc.L2::cache_hint.f64 %0, [%1], %2;" : "=d"(v) : "l"(p), "l"(policy));
    return v;
}
__device__ __forceinline__ void fence_proxy_async_smem() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

constexpr uint64_t kWaitLimitNs = 1000000000ull;   // 1 s per wait
constexpr uint64_t kDrainLimitNs = 100000000ull;   // 0.1 s per drain wait
constexpr int kErrTimeout = 6;                     // -SPMV_ETIMEOUT

__device__ __forceinline__ void store_row(const CsrArgs& a, int row, double sum) {
    if (a.rowmap) {
        const int o = __ldg(a.rowmap + row);
        a.y[o] = a.accumulate ? a.y[o] + sum : sum;
    } else {
        a.y[row] = a.accumulate ? a.y[row] + sum : sum;
    }
}

// ------------------------------------------------------------------------
// Pack: dst[k] = x[idx[k]] for every slot k (pos == nullptr) or for the
// slots listed in pos[0..count).  A thread takes kPackIlp slots a grid
// stride apart per step: their index loads, then their gathers, then their
// stores, so kPackIlp index-then-gather chains are in flight at once.  With
// `also` the same slots go to a second array, the receive buffer: pack and
// exchange in one launch, for streams of products through host buffers, whose
// operations follow one another (16 products of the 27-point stencil on 80^3
// 809 -> 772 us, on 20^3 245 -> 221 us; power-law 300 000 rows 1015 -> 983 us).
// Schedules keep a launch per operation: joining the two there changed nothing
// (replayed 64 x 64 grid 4.1 us and 150 000-row band matrix 8.7 us both ways).
// ------------------------------------------------------------------------
constexpr int kPackIlp = 4;

__global__ void __launch_bounds__(256) gather_kernel(const double* __restrict__ x,
                                                     const int32_t* __restrict__ idx,
                                                     const int32_t* __restrict__ pos,
                                                     double* __restrict__ dst, double* __restrict__ also,
                                                     int64_t count, int pdl) {
    pdl_begin(pdl);  // the previous kernel of this stream is done (unless independent)
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i0 < count; i0 += kPackIlp * stride) {
        int64_t k[kPackIlp];
        int32_t c[kPackIlp];
        double v[kPackIlp];
#pragma unroll
        for (int u = 0; u < kPackIlp; ++u) {
            const int64_t i = i0 + u * stride;
            k[u] = i < count ? (pos ? (int64_t)__ldg(pos + i) : i) : -1;
        }
#pragma unroll
        for (int u = 0; u < kPackIlp; ++u) c[u] = k[u] >= 0 ? __ldg(idx + k[u]) : 0;
#pragma unroll
        for (int u = 0; u < kPackIlp; ++u) v[u] = k[u] >= 0 ? __ldg(x + c[u]) : 0.0;
#pragma unroll
        for (int u = 0; u < kPackIlp; ++u)
            if (k[u] >= 0) {
                dst[k[u]] = v[u];
                if (also) also[k[u]] = v[u];
            }
    }
}

cudaError_t launch_gather(const double* x, const int32_t* idx, const int32_t* pos, double* dst, double* also,
                          int64_t count, int num_sms, cudaStream_t s, int pdl) {
    if (count <= 0) return cudaSuccess;
    int64_t blocks = (count + 256 * kPackIlp - 1) / (256 * kPackIlp);
    const int64_t cap = (int64_t)num_sms * 8;
    if (blocks > cap) blocks = cap;
    return launch_pdl(gather_kernel, dim3((unsigned)blocks), dim3(256), 0, s, x, idx, pos, dst, also, count,
                      pdl);
}

// ------------------------------------------------------------------------
// Halo exchange: dst[0..count) = src[0..count).  Aligned: 16-byte pairs,
// kPackIlp loads in flight per thread before their stores.
// ------------------------------------------------------------------------
__global__ void __launch_bounds__(256) copy_kernel(const double* __restrict__ src,
                                                   double* __restrict__ dst, int64_t count, int pdl) {
    pdl_begin(pdl);  // the previous kernel of this stream is done (unless independent)
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const bool vec = ((reinterpret_cast<uintptr_t>(src) | reinterpret_cast<uintptr_t>(dst)) & 15) == 0;
    if (vec) {
        const int64_t pairs = count >> 1;
        const double2* s2 = reinterpret_cast<const double2*>(src);
        double2* d2 = reinterpret_cast<double2*>(dst);
        for (int64_t i0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i0 < pairs; i0 += kPackIlp * stride) {
            double2 t[kPackIlp];
#pragma unroll
            for (int u = 0; u < kPackIlp; ++u)
                if (i0 + u * stride < pairs) t[u] = __ldg(s2 + i0 + u * stride);
#pragma unroll
            for (int u = 0; u < kPackIlp; ++u)
                if (i0 + u * stride < pairs) d2[i0 + u * stride] = t[u];
        }
        if ((count & 1) && blockIdx.x == 0 && threadIdx.x == 0) dst[count - 1] = src[count - 1];
    } else {
        for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += stride)
            dst[i] = __ldg(src + i);
    }
}

cudaError_t launch_copy(const double* src, double* dst, int64_t count, int num_sms,
                        cudaStream_t s, int pdl) {
    if (count <= 0) return cudaSuccess;
    int64_t blocks = (count / 2 + 256 * kPackIlp - 1) / (256 * kPackIlp);
    if (blocks < 1) blocks = 1;
    // 8 CTAs per SM: a 13 MB halo (a power-law rank's) in one round of loads
    // (3.8 us per rank against 4.2 us at 4 CTAs per SM; the 104 MB exchange
    // 32.5 us, 0.94 of the copy peak)
    const int64_t cap = (int64_t)num_sms * 8;
    if (blocks > cap) blocks = cap;
    return launch_pdl(copy_kernel, dim3((unsigned)blocks), dim3(256), 0, s, src, dst, count, pdl);
}

// ------------------------------------------------------------------------
// Thread-per-row CSR product over bulk-copied tiles (variants TILE and WARP).
//
// A tile is up to 32 consecutive rows of one rank and belongs to one warp,
// which copies the tile's values and columns (contiguous in the CSR) into its
// own stage of shared memory with two bulk copies against its own mbarrier
// (start addresses rounded down to 16 bytes, sizes rounded up; the device
// arrays are padded so the rounded reads stay in bounds).  Lane i sums row
// r0 + i in storage order with one DFMA per entry, U gathers of x in flight,
// into S sums: 1, or 2 (the entries at even and at odd places of the row, added
// at the end: half the chain of dependent FMAs, and a smaller rounding error).
// Warps never wait for each other.
//
// A tile whose entries do not fit the stage (TILE_WIDE) is summed the same
// way straight from global memory.  In a tile of TILE_LONG every row longer than
// kTileWarpRow is summed by the whole warp instead (lane l takes entries l, l+32,
// ..., then a fixed butterfly), so a long row costs its 32nd part.  A row longer
// than kTileCtaRow is a chain of too many rounds even for a warp and goes to a
// CTA (tile_row), in launches that have such rows (ROWS): their first CTAs take
// the rows, as many as the rows' share of the entries, the others the tiles.
// Each row is summed in a fixed order whatever the grid, the stream or the
// schedule, and no launch keeps anything for the next.
//
// What bounds it: HBM and the FP64 pipe once enough warps are resident, and
// the stages decide how many: one stage per warp, as large as 98 % of the
// plan's tiles need (27-point stencil: 864 entries, 10.4 KB, 20 warps per SM),
// where two stages of half as many warps or block-wide tiles of 128 rows took
// longer.  LOCAL products: 27-point 91^3 (19.9 M entries) 51 us against 77 us
// with block-wide double-buffered tiles and 71 us with two stages per warp;
// 7-point 120^3 33 us against 93 us; 27-point 20^3 4.5 us against 5.0 us.  Long
// rows are bound by their chains of load-then-gather rounds, so by how many warps
// share them: 400 rows of 20 000 entries 21 us (a warp for 32 of them in turn 2941
// us, block-wide tiles 41 us), 4000 of 3000 51 us (632 and 1426 us), one of
// 1 000 000 among 100 000 of 5 550 us (4439 and 592 us), power-law 1 M rows in one
// rank 143 us (160 us).
// ------------------------------------------------------------------------
constexpr int kTileWarpRow = 32;   // in a TILE_LONG tile, longer rows go to the whole warp
// warps per CTA: more for a row than for tiles, whose warps never wait for each other
template <bool ROWS>
constexpr int kTileCtaWarps = ROWS ? 8 : 4;

struct StageLayout {   // of one warp's stage for up to `cap` entries (a multiple of 32)
    int col_off, bytes;
    __host__ __device__ explicit StageLayout(int cap)
        : col_off((cap + 2) * 8), bytes((cap + 2) * 8 + (cap + 8) * 4) {}
};

// One row, entries [d.k0, d.k1), by the CTA: thread t takes entries t, t + T, ...
// (T threads, 8 of them in flight, the next columns loaded ahead), a fixed
// butterfly in each warp, then the warps' sums in warp order.
template <int WARPS>
__device__ __forceinline__ void tile_row(const CsrArgs& a, const Tile& d, uint64_t pol_keep) {
    constexpr int T = WARPS * 32, D = 8;
    __shared__ double s_part[WARPS];
    const unsigned n = (unsigned)(d.k1 - d.k0), t = threadIdx.x;   // unsigned: n + T D may pass 2^31
    const int32_t* col = a.col + d.k0;
    const double* val = a.val + d.k0;
    const double* xb = a.x + d.xoff;
    double part = 0.0;
    int32_t c[D];
#pragma unroll
    for (int u = 0; u < D; ++u) c[u] = t + T * u < n ? __ldg(col + t + T * u) : 0;
    for (unsigned base = 0; base < n; base += T * D) {
        const unsigned k = base + t;
        double vv[D], xv[D];
#pragma unroll
        for (int u = 0; u < D; ++u) {
            const bool m = k + T * u < n;
            xv[u] = m ? ldg_keep(xb + c[u], pol_keep) : 0.0;
            vv[u] = m ? __ldg(val + k + T * u) : 0.0;
        }
#pragma unroll
        for (int u = 0; u < D; ++u) c[u] = k + T * (D + u) < n ? __ldg(col + k + T * (D + u)) : 0;
#pragma unroll
        for (int u = 0; u < D; ++u) {
            const double p = fma(vv[u], xv[u], part);
            part = k + T * u < n ? p : part;
        }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) part += __shfl_xor_sync(0xffffffffu, part, off);
    if ((t & 31) == 0) s_part[t >> 5] = part;
    __syncthreads();
    if (t == 0) {
        double sum = s_part[0];
#pragma unroll
        for (int w = 1; w < WARPS; ++w) sum += s_part[w];
        store_row(a, d.r0, sum);
    }
    __syncthreads();   // s_part is rewritten for the next row
}

template <int U, int S, bool ROWS>
__global__ void __launch_bounds__(kTileCtaWarps<ROWS> * 32, (ROWS ? 4 : U > 9 ? 8 : 10))
    csr_tile_kernel(CsrArgs a, const Tile* __restrict__ tiles, int tile_begin, int tile_end, int cap,
                    const Tile* __restrict__ rows, int row_begin, int row_end, int row_ctas) {
    pdl_begin(a.pdl);  // the previous kernel of this stream is done (unless independent)
    static_assert(S == 1 || U % 2 == 0, "a round begins at an even place");
    constexpr int kTileWarps = kTileCtaWarps<ROWS>;
    const int cta = (int)blockIdx.x - (ROWS ? row_ctas : 0);   // among those that take tiles
    if (ROWS && cta < 0) {
        for (int r = row_begin + (int)blockIdx.x; r < row_end; r += row_ctas)
            tile_row<kTileWarps>(a, rows[r], policy_evict_last());
        return;
    }
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ __align__(8) uint64_t bars[kTileWarps];
    const uint64_t pol_stream = policy_evict_first();
    const uint64_t pol_keep = policy_evict_last();
    const int lane = threadIdx.x & 31;
    const int w = threadIdx.x >> 5;
    const StageLayout lay(cap);
    unsigned char* stage = smem + (size_t)w * lay.bytes;
    const double* vs = reinterpret_cast<const double*>(stage);
    const int32_t* cs = reinterpret_cast<const int32_t*>(stage + lay.col_off);
    const uint32_t bar = smem_u32(&bars[w]);
    if (lane == 0) {
        mbar_init(bar, 1);
        mbar_fence_init();
    }
    __syncwarp();
    uint32_t parity = 0;
    for (int t = tile_begin + cta * kTileWarps + w; t < tile_end; t += ((int)gridDim.x - (ROWS ? row_ctas : 0)) * kTileWarps) {
        const Tile d = tiles[t];
        const bool staged = d.flags == 0;
        const int va = d.k0 & ~1, ca = d.k0 & ~3;
        if (staged && lane == 0) {
            fence_proxy_async_smem();   // the stage was read by the warp before
            const uint32_t vbytes = (uint32_t)(((d.k1 + 1) & ~1) - va) * 8u;
            const uint32_t cbytes = (uint32_t)(((d.k1 + 3) & ~3) - ca) * 4u;
            mbar_arrive_expect_tx(bar, vbytes + cbytes);
            if (vbytes) bulk_g2s_hint(smem_u32(stage), a.val + va, vbytes, bar, pol_stream);
            if (cbytes) bulk_g2s_hint(smem_u32(stage + lay.col_off), a.col + ca, cbytes, bar, pol_stream);
        }
        const int row = d.r0 + lane;
        const bool live = row < d.r1;
        const int kb = live ? __ldg(a.ptr + row) : 0;
        const int len = live ? __ldg(a.ptr + row + 1) - kb : 0;
        const double* xb = a.x + d.xoff;
        const int warp_row = d.flags & TILE_LONG ? kTileWarpRow : INT32_MAX;
        const bool mine = len <= warp_row;
        const int cnt = mine ? len : 0;
        const int wmax = __reduce_max_sync(0xffffffffu, cnt);
        double sum[2] = {0.0, 0.0};
        if (staged) {
            const bool ok = mbar_wait_bounded(bar, parity, kWaitLimitNs);
            if (__any_sync(0xffffffffu, !ok)) {
                if (lane == 0) {   // let the copies still in flight land before the warp leaves
                    atomicExch(a.err, kErrTimeout);
                    mbar_wait_bounded(bar, parity, kDrainLimitNs);
                }
                break;
            }
            parity ^= 1;
        }
        // gathers in flight before their FMAs; slots past the row read x[xoff]
        // (a valid address), and their FMA results are discarded; FMAs run in
        // storage order
        if (staged) {
            const double* vr = vs + (kb - va);
            const int32_t* cr = cs + (kb - ca);
            for (int base = 0; base < wmax; base += U) {
                double xv[U];
#pragma unroll
                for (int u = 0; u < U; ++u) xv[u] = ldg_keep(xb + (base + u < cnt ? cr[base + u] : 0), pol_keep);
#pragma unroll
                for (int u0 = 0; u0 < U; u0 += 3) {   // values three at a time, ahead of the dependent FMAs
                    double vv[3];
#pragma unroll
                    for (int i = 0; i < 3; ++i) vv[i] = u0 + i < U && base + u0 + i < cnt ? vr[base + u0 + i] : 0.0;
#pragma unroll
                    for (int i = 0; i < 3 && u0 + i < U; ++i) {
                        if (base + u0 + i >= wmax) break;   // warp-uniform
                        double& acc = sum[(u0 + i) % S];
                        const double p = fma(vv[i], xv[u0 + i], acc);
                        acc = base + u0 + i < cnt ? p : acc;
                    }
                }
            }
        } else {
#pragma unroll 1
            for (int base = 0; base < wmax; base += 4) {
                double xv[4], vv[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const bool m = base + u < cnt;
                    vv[u] = m ? __ldg(a.val + kb + base + u) : 0.0;
                    xv[u] = ldg_keep(xb + (m ? __ldg(a.col + kb + base + u) : 0), pol_keep);
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    double& acc = sum[u % S];
                    const double p = fma(vv[u], xv[u], acc);
                    acc = base + u < cnt ? p : acc;
                }
            }
        }
        if (live && mine) store_row(a, row, S == 2 ? sum[0] + sum[1] : sum[0]);
        for (unsigned todo = __ballot_sync(0xffffffffu, !mine); todo; todo &= todo - 1) {
            const int src = __ffs(todo) - 1;
            const int k0 = __shfl_sync(0xffffffffu, kb, src), n = __shfl_sync(0xffffffffu, len, src);
            double part = 0.0;
#pragma unroll 1
            for (int k = lane; k - lane < n; k += 32 * 4) {
                double xv[4], vv[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const bool m = k + 32 * u < n;
                    vv[u] = m ? __ldg(a.val + k0 + k + 32 * u) : 0.0;
                    xv[u] = m ? ldg_keep(xb + __ldg(a.col + k0 + k + 32 * u), pol_keep) : 0.0;
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    if (k - lane + 32 * u >= n) break;   // warp-uniform
                    const double p = fma(vv[u], xv[u], part);
                    part = k + 32 * u < n ? p : part;
                }
            }
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) part += __shfl_xor_sync(0xffffffffu, part, off);
            if (lane == 0) store_row(a, d.r0 + src, part);
        }
        __syncwarp();   // the stage is free again
    }
}

int tile_stage_cap(int entries) {
    const int cap = (entries + 31) / 32 * 32;
    return cap < 64 ? 64 : cap > kTileMaxEntries ? kTileMaxEntries : cap;
}

template <int U, int S, bool ROWS>
static cudaError_t run_tile(const CsrArgs& a, const TileSpan& t, int num_sms, cudaStream_t s) {
    constexpr int kTileWarps = kTileCtaWarps<ROWS>;
    const size_t smem = (size_t)kTileWarps * StageLayout(t.cap).bytes;
    static std::atomic<unsigned long long> configured{0};   // one bit per device ordinal
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev >= 64 || !(configured.load(std::memory_order_acquire) >> dev & 1ull)) {
        e = cudaFuncSetAttribute(csr_tile_kernel<U, S, ROWS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 kTileWarps * StageLayout(kTileMaxEntries).bytes);
        if (e != cudaSuccess) return e;
        if (dev < 64) configured.fetch_or(1ull << dev, std::memory_order_acq_rel);
    }
    // CTAs per SM by stage size (a query costs the host about a microsecond)
    static std::atomic<int> known[kTileMaxEntries / 32 + 1];
    int occ = dev == 0 ? known[t.cap / 32].load(std::memory_order_relaxed) : 0;
    if (occ == 0) {
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, csr_tile_kernel<U, S, ROWS>, kTileWarps * 32, smem);
        if (e != cudaSuccess) return e;
        if (occ < 1) return cudaErrorInvalidConfiguration;
        if (dev == 0) known[t.cap / 32].store(occ, std::memory_order_relaxed);
    }
    const int most = num_sms * occ, need = (t.end - t.begin + kTileWarps - 1) / kTileWarps;
    int row_ctas = 0;
    if (ROWS) {
        row_ctas = need > 0 ? std::min(std::max((int)(t.row_share * most), 1), most - 1) : most;
        row_ctas = std::min(row_ctas, t.row_end - t.row_begin);
    }
    const int grid = row_ctas + std::min(need, most - row_ctas);
    return launch_pdl(csr_tile_kernel<U, S, ROWS>, dim3(grid), dim3(kTileWarps * 32), smem, s, a, t.tiles,
                      t.begin, t.end, t.cap, t.rows, t.row_begin, t.row_end, row_ctas);
}

bool tile_param_supported(int param) { return param >= 0 && param < 5; }

// Geometries: gathers in flight per lane.  TILE keeps two sums a row (geometry
// 3: one), WARP one.
cudaError_t launch_tile(const CsrArgs& a, const TileSpan& t, bool one_sum, int param, int num_sms, cudaStream_t s) {
    const bool rows = t.row_end > t.row_begin;
#define TILE_RUN(u, sums) return rows ? run_tile<u, sums, true>(a, t, num_sms, s) : run_tile<u, sums, false>(a, t, num_sms, s)
    switch (one_sum ? param + 5 : param) {
        case 0: TILE_RUN(8, 2);
        case 1: TILE_RUN(14, 2);
        case 2: TILE_RUN(4, 2);
        case 4: TILE_RUN(16, 2);
        case 5: TILE_RUN(9, 1);
        case 6: TILE_RUN(14, 1);
        case 7: TILE_RUN(4, 1);
        case 3:
        case 8: TILE_RUN(7, 1);
        case 9: TILE_RUN(16, 1);
        default: return cudaErrorInvalidValue;
    }
#undef TILE_RUN
}

// ------------------------------------------------------------------------
// Vector-per-row CSR: V lanes share a row; each lane reads 4 consecutive
// entries per step with 128-bit loads (two double2 values, one int4 of
// columns) from a 4-aligned start, masks entries outside the row, and the
// V partial sums meet in a fixed xor-butterfly.  Rows come from the same
// tile table (rows r0..r1 with their x offset).
// ------------------------------------------------------------------------
template <int V>
__global__ void __launch_bounds__(256) csr_vector_kernel(CsrArgs a, const Tile* __restrict__ tiles,
                                                         int tile_begin, int tile_end) {
    pdl_begin(a.pdl);  // the previous kernel of this stream is done (unless independent)
    constexpr int GROUPS = 256 / V;
    const uint64_t pol_keep = policy_evict_last();
    const int lane = threadIdx.x % V;
    const int group = threadIdx.x / V;
    for (int t = tile_begin + (int)blockIdx.x; t < tile_end; t += (int)gridDim.x) {
        const Tile d = tiles[t];
        const double* xb = a.x + d.xoff;
        for (int rbase = d.r0; rbase < d.r1; rbase += GROUPS) {
            const int row = rbase + group;
            double sum = 0.0;
            if (row < d.r1) {
                // unsigned: the step past the last entry may pass 2^31
                const unsigned kb = __ldg(a.ptr + row), ke = __ldg(a.ptr + row + 1);
                for (unsigned k4 = (kb & ~3u) + 4 * lane; k4 < ke; k4 += 4 * V) {
                    const int4 c = __ldg(reinterpret_cast<const int4*>(a.col + k4));
                    const double2 v0 = __ldg(reinterpret_cast<const double2*>(a.val + k4));
                    const double2 v1 = __ldg(reinterpret_cast<const double2*>(a.val + k4 + 2));
                    const bool m0 = k4 + 0 >= kb && k4 + 0 < ke, m1 = k4 + 1 >= kb && k4 + 1 < ke;
                    const bool m2 = k4 + 2 >= kb && k4 + 2 < ke, m3 = k4 + 3 >= kb && k4 + 3 < ke;
                    // masked slots read x[xoff]: entries of a neighbouring
                    // row may index another rank's block
                    const double x0 = ldg_keep(xb + (m0 ? c.x : 0), pol_keep);
                    const double x1 = ldg_keep(xb + (m1 ? c.y : 0), pol_keep);
                    const double x2 = ldg_keep(xb + (m2 ? c.z : 0), pol_keep);
                    const double x3 = ldg_keep(xb + (m3 ? c.w : 0), pol_keep);
                    double t;
                    t = fma(v0.x, x0, sum); sum = m0 ? t : sum;
                    t = fma(v0.y, x1, sum); sum = m1 ? t : sum;
                    t = fma(v1.x, x2, sum); sum = m2 ? t : sum;
                    t = fma(v1.y, x3, sum); sum = m3 ? t : sum;
                }
            }
#pragma unroll
            for (int off = V / 2; off > 0; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off, V);
            if (row < d.r1 && lane == 0) store_row(a, row, sum);
        }
    }
}

// ------------------------------------------------------------------------
// Pair-per-lane CSR: V lanes share a row; the row's entries are covered by
// aligned pairs [k, k+1) (k even) and lane h takes pairs h, h+V, h+2V, ...
// Each pair is one 16-byte load of values and one 8-byte load of columns.
// FP64 cost on this part is per warp instruction whatever the active mask,
// so the FMA loop runs exactly as many pairs as the warp's longest share
// (warp-uniform), U pairs of gathers are in flight per lane, and the V
// partial sums meet in a fixed xor-butterfly.  For a 27-entry row and V = 2
// this is 14 FMA instructions + 1 add per 16 rows.
// ------------------------------------------------------------------------
template <int V, int U, int MINB>
__global__ void __launch_bounds__(256, MINB) csr_pair_kernel(CsrArgs a, const Tile* __restrict__ tiles,
                                                          int tile_begin, int tile_end) {
    pdl_begin(a.pdl);  // the previous kernel of this stream is done (unless independent)
    constexpr int GROUPS = 256 / V;
    const uint64_t pol_keep = policy_evict_last();
    const int lane = threadIdx.x % V;
    const int group = threadIdx.x / V;
    for (int t = tile_begin + (int)blockIdx.x; t < tile_end; t += (int)gridDim.x) {
        const Tile d = tiles[t];
        const double* xb = a.x + d.xoff;
        for (int rbase = d.r0; rbase < d.r1; rbase += GROUPS) {
            const int row = rbase + group;
            int kb = 0, ke = 0, k2 = 0, cnt = 0;
            if (row < d.r1) {
                kb = __ldg(a.ptr + row);
                ke = __ldg(a.ptr + row + 1);
                k2 = kb & ~1;
                const int npairs = (ke - k2 + 1) >> 1;
                cnt = npairs > lane ? (npairs - lane + V - 1) / V : 0;
            }
            const int wmax = __reduce_max_sync(0xffffffffu, cnt);
            double sum = 0.0;
            for (int j0 = 0; j0 < wmax; j0 += U) {
                double2 vv[U];
                double x0[U], x1[U];
                bool m0[U], m1[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int j = j0 + u;
                    const bool act = j < cnt;
                    const int k = act ? k2 + 2 * (lane + V * j) : k2;   // k2 is a valid even index
                    vv[u] = __ldg(reinterpret_cast<const double2*>(a.val + k));
                    const int2 c = __ldg(reinterpret_cast<const int2*>(a.col + k));
                    m0[u] = act && k >= kb;
                    m1[u] = act && k + 1 < ke;
                    x0[u] = ldg_keep(xb + (m0[u] ? c.x : 0), pol_keep);
                    x1[u] = ldg_keep(xb + (m1[u] ? c.y : 0), pol_keep);
                }
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    if (j0 + u >= wmax) break;   // warp-uniform
                    double t0 = fma(vv[u].x, x0[u], sum);
                    sum = m0[u] ? t0 : sum;
                    t0 = fma(vv[u].y, x1[u], sum);
                    sum = m1[u] ? t0 : sum;
                }
            }
#pragma unroll
            for (int off = V / 2; off > 0; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off, V);
            if (row < d.r1 && lane == 0) store_row(a, row, sum);
        }
    }
}

cudaError_t launch_pairs(const CsrArgs& a, const Tile* tiles, int tile_begin, int tile_end, int lanes,
                         int num_sms, cudaStream_t s) {
    if (tile_end <= tile_begin) return cudaSuccess;
    int grid = num_sms * 8;
    if (grid > tile_end - tile_begin) grid = tile_end - tile_begin;
    // lanes 1/2/4/8: 4 pairs in flight per lane (up to 64 registers);
    // 102/104: 2 or 4 lanes with 2 pairs in flight in 32 registers, so 8
    // CTAs (64 warps) fit on an SM
    cudaError_t e = cudaSuccess;
    switch (lanes) {
        case 1: e = launch_pdl(csr_pair_kernel<1, 4, 4>, dim3(grid), dim3(256), 0, s, a, tiles, tile_begin, tile_end); break;
        case 2: e = launch_pdl(csr_pair_kernel<2, 4, 4>, dim3(grid), dim3(256), 0, s, a, tiles, tile_begin, tile_end); break;
        case 4: e = launch_pdl(csr_pair_kernel<4, 4, 4>, dim3(grid), dim3(256), 0, s, a, tiles, tile_begin, tile_end); break;
        case 8: e = launch_pdl(csr_pair_kernel<8, 2, 4>, dim3(grid), dim3(256), 0, s, a, tiles, tile_begin, tile_end); break;
        case 102: e = launch_pdl(csr_pair_kernel<2, 2, 8>, dim3(grid), dim3(256), 0, s, a, tiles, tile_begin, tile_end); break;
        case 104: e = launch_pdl(csr_pair_kernel<4, 2, 8>, dim3(grid), dim3(256), 0, s, a, tiles, tile_begin, tile_end); break;
        default: return cudaErrorInvalidValue;
    }
    return e;
}

cudaError_t launch_vector(const CsrArgs& a, const Tile* tiles, int tile_begin, int tile_end,
                          int lanes, int num_sms, cudaStream_t s) {
    if (tile_end <= tile_begin) return cudaSuccess;
    int grid = num_sms * 8;
    if (grid > tile_end - tile_begin) grid = tile_end - tile_begin;
    cudaError_t e = cudaSuccess;
    switch (lanes) {
        case 2: e = launch_pdl(csr_vector_kernel<2>, dim3(grid), dim3(256), 0, s, a, tiles, tile_begin, tile_end); break;
        case 4: e = launch_pdl(csr_vector_kernel<4>, dim3(grid), dim3(256), 0, s, a, tiles, tile_begin, tile_end); break;
        case 8: e = launch_pdl(csr_vector_kernel<8>, dim3(grid), dim3(256), 0, s, a, tiles, tile_begin, tile_end); break;
        case 16: e = launch_pdl(csr_vector_kernel<16>, dim3(grid), dim3(256), 0, s, a, tiles, tile_begin, tile_end); break;
        case 32: e = launch_pdl(csr_vector_kernel<32>, dim3(grid), dim3(256), 0, s, a, tiles, tile_begin, tile_end); break;
        default: return cudaErrorInvalidValue;
    }
    return e;
}

// ------------------------------------------------------------------------
// Self-test of the bounded wait: one thread waits on an mbarrier that no
// copy and no thread ever completes; the wait gives up after limit_ns and
// the kernel reports SPMV_ETIMEOUT's magnitude through `status`.
// ------------------------------------------------------------------------
__global__ void selftest_wait_kernel(uint64_t limit_ns, int* status) {
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(smem_u32(&bar), 1);
        mbar_fence_init();
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        const bool ok = mbar_wait_bounded(smem_u32(&bar), 0u, limit_ns);
        *status = ok ? 0 : kErrTimeout;
    }
}

cudaError_t selftest_wait_timeout(uint64_t limit_ns, int* status_host) {
    int* d = nullptr;
    cudaError_t e = cudaMalloc(&d, sizeof(int));
    if (e != cudaSuccess) return e;
    selftest_wait_kernel<<<1, 32>>>(limit_ns, d);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpy(status_host, d, sizeof(int), cudaMemcpyDeviceToHost);
    cudaFree(d);
    return e;
}

// ------------------------------------------------------------------------
// FP64 FMA throughput probe: the first `lanes` lanes of every warp run 8
// independent chains of `iters` fused multiply-adds each (enough chains to
// cover the pipe's latency), then store their sum, so no chain is dead code.
// Each chain accumulates through the addend, a = fma(m, c, a), as a product
// accumulates sum = fma(value, x, sum), with every operand a register of its
// own (m and c pass through an opaque move, so they are not folded into
// constant operands).  m c = 1e-6 keeps every value near 1 (no overflow, no
// subnormals).
// ------------------------------------------------------------------------
constexpr int kProbeThreads = 256;
constexpr int kProbeChains = 8;

__device__ __forceinline__ double opaque(double v) {
    double r;
    asm volatile("mov.b64 %0, %1;" : "=d"(r) : "d"(v));
    return r;
}

__global__ void __launch_bounds__(kProbeThreads) dfma_probe_kernel(int64_t iters, int lanes, double* out) {
    const int64_t gid = (int64_t)blockIdx.x * kProbeThreads + threadIdx.x;
    double a[kProbeChains], m[kProbeChains], c[kProbeChains];
#pragma unroll
    for (int u = 0; u < kProbeChains; ++u) {
        a[u] = 1.0 + 1e-3 * u + 1e-9 * (double)(gid & 1023);
        m[u] = opaque(1e-3);
        c[u] = opaque(1e-3);
    }
    if ((int)(threadIdx.x & 31) < lanes) {
        for (int64_t i = 0; i < iters; ++i) {
#pragma unroll
            for (int u = 0; u < kProbeChains; ++u) a[u] = fma(m[u], c[u], a[u]);
        }
    }
    double sum = 0.0;
#pragma unroll
    for (int u = 0; u < kProbeChains; ++u) sum += a[u];
    out[gid] = sum;
}

int probe_threads() { return kProbeThreads; }

cudaError_t launch_dfma_probe(int64_t iters, int grid, int lanes, double* out, int64_t* dfma, cudaStream_t s) {
    dfma_probe_kernel<<<grid, kProbeThreads, 0, s>>>(iters, lanes, out);
    *dfma = (int64_t)grid * (kProbeThreads / 32) * lanes * kProbeChains * iters;
    return cudaGetLastError();
}

// ------------------------------------------------------------------------
// Gather throughput probe: thread g of T sums table[idx[k]] over k = g,
// g + T, g + 2T, ... (four gathers in flight), the access pattern of a
// product's x gathers with the column stream read coalesced; each thread
// stores its sum.
// ------------------------------------------------------------------------
__global__ void __launch_bounds__(kProbeThreads) gather_probe_kernel(const double* __restrict__ table,
                                                                     const int32_t* __restrict__ idx,
                                                                     int64_t count, double* out) {
    const int64_t T = (int64_t)gridDim.x * kProbeThreads;
    const int64_t g = (int64_t)blockIdx.x * kProbeThreads + threadIdx.x;
    double sum = 0.0;
    int64_t k = g;
    for (; k + 3 * T < count; k += 4 * T) {
        const int32_t i0 = __ldg(idx + k), i1 = __ldg(idx + k + T), i2 = __ldg(idx + k + 2 * T),
                      i3 = __ldg(idx + k + 3 * T);
        const double v0 = __ldg(table + i0), v1 = __ldg(table + i1), v2 = __ldg(table + i2),
                     v3 = __ldg(table + i3);
        sum += v0;
        sum += v1;
        sum += v2;
        sum += v3;
    }
    for (; k < count; k += T) sum += __ldg(table + __ldg(idx + k));
    out[g] = sum;
}

cudaError_t launch_gather_probe(const double* table, const int32_t* idx, int64_t count, int grid, double* out,
                                cudaStream_t s) {
    gather_probe_kernel<<<grid, kProbeThreads, 0, s>>>(table, idx, count, out);
    return cudaGetLastError();
}

}  // namespace spmvk
