// Merge-path CSR product for skewed row lengths (the K-merge kernel).
//
// The rows' end offsets and the entry indices are merged into one path of
// rows + entries items (Merrill and Garland's merge-based CSR), and every
// warp takes a range of the path, so all do the same work however long the
// rows are.  A warp walks its entries 256 at a time, eight consecutive ones a
// lane: 32-byte loads, eight x gathers in flight, eight FMAs.  Rows that end
// within a lane's entries are told by byte flags in shared memory, which the
// lanes that hold the row ends set; a row cut between lanes is finished by a
// segmented scan over the lanes, one cut between chunks by the warp's running
// partial, one cut between warps by a carry that a second kernel adds in range
// order.  No atomics and no data-dependent order: results depend only on the
// matrix.
//
// What bounds it: the scattered x gathers (38 us for 10.8 M at the rate of
// random reads) and the FP64 pipe (about 14 FP64 instructions per 8 entries of
// a lane; 0.70 of the pipe's active cycles on 28.6 M entries).  Power-law matrix
// of 700 001 rows, 10.8 M entries: 68 us (70 us with 16-byte loads); the form
// before, tiles of 2048 items staged in shared memory per CTA and walked item by
// item (48 M warp instructions against 19 M, 24 warps per SM, a path search of 22
// dependent shared-memory reads a thread, and a launch of its own that computed
// the tiles), took 154 us.  7-point stencil of 12 696 rows: 6.2 us against 14.3 us.
#include "internal.h"
#include "merge_chunks.h"
#include "pdl.cuh"

#include <cuda_runtime.h>

#include <mutex>

namespace spmvk {

// Error word of launches that have no plan (CsrArgs::err == nullptr).
__device__ int g_csr_err = 0;

namespace {

constexpr int MERGE_NT = 256;                 // threads per CTA
constexpr int MERGE_WARPS = MERGE_NT / 32;
constexpr int kErrTimeout = 6;

// Items per range.  A chunk starts at a multiple of MERGE_LANE entries, so a
// range of MERGE_CHUNK m - MERGE_LANE items never needs more than m chunks.
// Plans use one chunk while that makes at most two ranges for every warp in
// flight, else two; plan-free products the length that gives 4864 ranges
// (152 SMs x 32 warps: one wave of equal ranges), at least one chunk.  It
// depends on the matrix alone, so results do too.
// One chunk against two, replayed schedules of per-rank / whole launches (us):
// band matrix of 22 760 rows 20.8 / 10.8 against 26.6 / 13.3, of 200 000 rows
// (2.2 M items) 30.6 / 22.4 against 33.5 / 21.9, 7-point stencil on 60^3 24.4 /
// 15.1 against 27.4 / 15.4; above the line power-law 1 M rows 156 / 111 against
// 143 / 110, 27-point on 91^3 101 / 85.6 against 99.7 / 83.4.
constexpr int MERGE_RANGES = 4864;

int64_t range_items(int64_t items) {
    const int64_t per = (items + MERGE_RANGES - 1) / MERGE_RANGES;
    const int64_t chunks = (per + MERGE_LANE + MERGE_CHUNK - 1) / MERGE_CHUNK;
    return MERGE_CHUNK * chunks - MERGE_LANE;
}

// Merge-path coordinate of diagonal d in the merge of row ends A[0..a_len)
// (A[i] = end of row i minus the entry base) with entry indices 0..b_len:
// returns the number of row ends consumed.  Row end i precedes entry j
// when A[i] <= j.
template <class F>
__device__ __forceinline__ int path_search(int d, int a_len, int b_len, F A) {
    int lo = d - b_len > 0 ? d - b_len : 0;
    int hi = d < a_len ? d : a_len;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (A(mid) <= d - mid - 1) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

// The same for two diagonals at once by the whole warp: 32 probes of each per
// step, so n rows take log32(n) dependent reads instead of log2(n).
template <class F>
__device__ __forceinline__ void warp_path_search(int d0, int d1, int a_len, int b_len, F A, int& i0, int& i1) {
    const int lane = threadIdx.x & 31;
    int lo0 = d0 - b_len > 0 ? d0 - b_len : 0, hi0 = d0 < a_len ? d0 : a_len;
    int lo1 = d1 - b_len > 0 ? d1 - b_len : 0, hi1 = d1 < a_len ? d1 : a_len;
    while (lo0 < hi0 || lo1 < hi1) {   // both are the same in every lane
        const int s0 = (hi0 - lo0 + 31) >> 5, s1 = (hi1 - lo1 + 31) >> 5;
        const int p0 = lo0 + (lane + 1) * s0 - 1, p1 = lo1 + (lane + 1) * s1 - 1;
        const bool t0 = s0 > 0 && p0 < hi0 && A(p0) <= d0 - p0 - 1;
        const bool t1 = s1 > 0 && p1 < hi1 && A(p1) <= d1 - p1 - 1;
        const int n0 = __popc(__ballot_sync(0xffffffffu, t0)), n1 = __popc(__ballot_sync(0xffffffffu, t1));
        if (s0 > 0) {   // the first probe that fails bounds the answer
            lo0 += n0 * s0;
            hi0 = hi0 < lo0 + s0 - 1 ? hi0 : lo0 + s0 - 1;
        }
        if (s1 > 0) {
            lo1 += n1 * s1;
            hi1 = hi1 < lo1 + s1 - 1 ? hi1 : lo1 + s1 - 1;
        }
    }
    i0 = lo0;
    i1 = lo1;
}

__device__ __forceinline__ void put(const CsrArgs& a, int row, double v) {
    const int o = a.rowmap ? __ldg(a.rowmap + row) : row;
    a.y[o] = a.accumulate ? a.y[o] + v : v;
}

// Range t = blockIdx.x * 8 + warp (grid-stride up to the launch's last).
// PLAN: ranges come from the plan's table, whose arrays are padded past their
// ends.  Else the warp finds its range of `items` merge items by itself, and
// the arrays are the caller's: the vector loads stop at the last entry.
// A32: values and columns start at multiples of 32 bytes (a plan's do), so a
// lane's entries are three 32-byte loads instead of six of 16 bytes.
template <bool PLAN, bool A32>
__global__ void __launch_bounds__(MERGE_NT, 4) merge_kernel(CsrArgs a, const MergeTile* __restrict__ tiles,
                                                            int tile_begin, int tile_end, int items,
                                                            Carry* __restrict__ carries) {
    // the previous kernel of this stream is done (unless independent); the
    // next kernel is this operation's fixup, which waits for the carries and
    // may be placed as CTAs leave
    pdl_begin((a.pdl & kPdlNoWait) | kPdlEarly);
    __shared__ __align__(16) unsigned char s_flag[MERGE_WARPS][MERGE_CHUNK];   // entry ends a row
    __shared__ double s_tot[MERGE_WARPS][MERGE_CHUNK];                         // total of the row that ends there
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned char* flag = s_flag[warp];
    double* tot = s_tot[warp];
    uint2* const my_flags = reinterpret_cast<uint2*>(flag + MERGE_LANE * lane);
    *my_flags = make_uint2(0u, 0u);
    __syncwarp();
    for (int t = tile_begin + (int)blockIdx.x * MERGE_WARPS + warp; t < tile_end; t += (int)gridDim.x * MERGE_WARPS) {
        if (a.abort_tile > 0 && t >= a.abort_tile - 1) {   // test hook
            if (lane == 0) {
                atomicExch(a.err ? a.err : &g_csr_err, kErrTimeout);
                carries[t] = Carry{-1, 0, 0.0};
            }
            continue;
        }
        // rows [r0, r1) end in the range, entries [k0, k1) lie in it
        int r0, r1, k0, k1;
        const double* xb = a.x;
        if (PLAN) {
            const MergeTile d = tiles[t];
            r0 = d.r0;
            r1 = d.r1;
            k0 = d.k0;
            k1 = d.k1;
            xb += d.xoff;
        } else {
            const int64_t all = (int64_t)a.n_rows + a.nnz_total;
            const int64_t e0 = (int64_t)t * items, e1 = e0 + items;
            const int d0 = (int)e0, d1 = (int)(e1 < all ? e1 : all);
            warp_path_search(d0, d1, a.n_rows, a.nnz_total, [&](int i) { return __ldg(a.ptr + i + 1); }, r0, r1);
            k0 = d0 - r0;
            k1 = d1 - r1;
        }
        int cur = r0;          // first row whose end has not been passed
        double open = 0.0;     // partial sum of row `cur` over the chunks so far
        for (unsigned c = merge_first_chunk(k0); c < (unsigned)k1; c += MERGE_CHUNK) {
            const unsigned e = c + MERGE_LANE * lane;
            double v[MERGE_LANE];
            int32_t col[MERGE_LANE];
            if (e < (unsigned)k1 && (PLAN || e + MERGE_LANE <= (unsigned)a.nnz_total)) {
                if (A32) {
                    asm("ld.global.nc.v8.s32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                        : "=r"(col[0]), "=r"(col[1]), "=r"(col[2]), "=r"(col[3]), "=r"(col[4]), "=r"(col[5]),
                          "=r"(col[6]), "=r"(col[7])
                        : "l"(a.col + e));
#pragma unroll
                    for (int u = 0; u < MERGE_LANE; u += 4)
                        asm("ld.global.nc.v4.f64 {%0, %1, %2, %3}, [%4];"
                            : "=d"(v[u]), "=d"(v[u + 1]), "=d"(v[u + 2]), "=d"(v[u + 3])
                            : "l"(a.val + e + u));
                } else {
                    const int4 c0 = __ldg(reinterpret_cast<const int4*>(a.col + e));
                    const int4 c1 = __ldg(reinterpret_cast<const int4*>(a.col + e + 4));
                    col[0] = c0.x; col[1] = c0.y; col[2] = c0.z; col[3] = c0.w;
                    col[4] = c1.x; col[5] = c1.y; col[6] = c1.z; col[7] = c1.w;
#pragma unroll
                    for (int u = 0; u < MERGE_LANE; u += 2) {
                        const double2 p = __ldg(reinterpret_cast<const double2*>(a.val + e + u));
                        v[u] = p.x;
                        v[u + 1] = p.y;
                    }
                }
            } else {
#pragma unroll
                for (int u = 0; u < MERGE_LANE; ++u) {
                    const bool in = e + u < (unsigned)k1;
                    col[u] = in ? __ldg(a.col + e + u) : 0;
                    v[u] = in ? __ldg(a.val + e + u) : 0.0;
                }
            }
            double xv[MERGE_LANE];
#pragma unroll
            for (int u = 0; u < MERGE_LANE; ++u) {
                const bool in = merge_in_range(e + u, k0, k1);   // neighbours of the range's first and last entries
                xv[u] = in ? __ldg(xb + col[u]) : 0.0;
                v[u] = in ? v[u] : 0.0;
            }
            // flag the last entry of every row that ends in the chunk and has
            // an entry in the range
            int row = cur;
            for (;;) {
                const int r = row + lane;
                const int end = r < r1 ? __ldg(a.ptr + r + 1) : 0;
                const bool here = r < r1 && merge_ends_by(end, c);
                if (here) {
                    const int beg = __ldg(a.ptr + r);
                    if (end > (beg > k0 ? beg : k0)) flag[end - 1 - c] = 1;
                }
                const int n = __popc(__ballot_sync(0xffffffffu, here));
                row += n;
                if (n < 32) break;
            }
            __syncwarp();
            const uint2 fl = *my_flags;
            *my_flags = make_uint2(0u, 0u);
            const bool any = (fl.x | fl.y) != 0;
            // the lane's entries in order; the first row that ends here may
            // have begun in earlier lanes
            double acc = 0.0, head = 0.0;
            int at = -1;
#pragma unroll
            for (int u = 0; u < MERGE_LANE; ++u) {
                acc = fma(v[u], xv[u], acc);
                if (((u < 4 ? fl.x : fl.y) >> (8 * (u & 3))) & 1u) {
                    if (at < 0) {
                        at = MERGE_LANE * lane + u;
                        head = acc;
                    } else {
                        tot[MERGE_LANE * lane + u] = acc;
                    }
                    acc = 0.0;
                }
            }
            // acc: what the lane adds to the row still open after it; sums over
            // the lanes since the last row end, in a fixed order
            const unsigned ends = __ballot_sync(0xffffffffu, any);
            const unsigned before = ends & ((2u << lane) - 1u);
            const int reach = before ? lane - (31 - __clz(before)) : lane;   // lanes that may be added
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                if (!__any_sync(0xffffffffu, off <= reach)) break;
                const double up = __shfl_up_sync(0xffffffffu, acc, off);
                if (off <= reach) acc = up + acc;
            }
            const double prev = __shfl_up_sync(0xffffffffu, acc, 1);
            if (any) {
                if (lane > 0) head = prev + head;
                if ((ends & ((1u << lane) - 1u)) == 0) head = open + head;
                tot[at] = head;
            }
            const double last = __shfl_sync(0xffffffffu, acc, 31);
            open = ends ? last : open + last;
            __syncwarp();
            for (int r = cur + lane; r < row; r += 32) {
                const int beg = __ldg(a.ptr + r), end = __ldg(a.ptr + r + 1);
                put(a, r, end > (beg > k0 ? beg : k0) ? tot[end - 1 - c] : 0.0);
            }
            cur = row;
            __syncwarp();   // tot is rewritten by the next chunk
        }
        for (int r = cur + lane; r < r1; r += 32) put(a, r, 0.0);   // a range without entries
        if (lane == 0) {
            Carry cy{-1, 0, 0.0};
            if (r1 < a.n_rows && k1 > k0) {
                const int beg = __ldg(a.ptr + r1);
                if (k1 > (beg > k0 ? beg : k0)) cy = Carry{r1, 0, open};
            }
            carries[t] = cy;
        }
    }
}

// Adds the ranges' carries to their rows: the first range of each run of
// ranges carrying the same row sums the run and adds it once.  A thread adds its
// run's next eight carries at once, then eight more, and goes on while more than
// two runs that begin in its warp's 32 ranges do; one or two, which may go on for
// thousands of ranges, are added by the whole warp: lane l takes every 32nd carry,
// eight in flight, then a fixed butterfly.  One row of 1 000 000 entries, product
// with 100 000 rows of 5: plan 27 us, plan-free 22 us, against 307 and 160 us with
// a thread summing every run (77 and 84 us with an eighth of the ranges); one of
// 10 000 11.9 and 12.6 us (12.3 and 13.0, 10.8 and 19.4 us); power-law 700 001 rows
// 68 us either way.
__global__ void __launch_bounds__(256) merge_fixup_kernel(CsrArgs a, const Carry* __restrict__ carries,
                                                          int tile_begin, int tile_end) {
    pdl_begin(a.pdl & kPdlEarly);   // the carries of the merge kernel are complete
    const int lane = threadIdx.x & 31;
    const int t = tile_begin + (int)(blockIdx.x * blockDim.x + threadIdx.x);
    auto carry = [&](int u) { return u < tile_end ? carries[u] : Carry{-1, 0, 0.0}; };
    const Carry c = carry(t);
    // a carry of a row of this product, the first of its run
    const bool first = c.row >= 0 && c.row < a.n_rows && (t == tile_begin || carries[t - 1].row != c.row);
    double tot = c.val;
    int u = t + 1;   // the next carry of the run, if it goes on
    bool on = first;
    int runs = 32;   // runs of the warp that go on
    for (int round = 0; runs > (round < 2 ? 0 : 2); ++round) {
        if (on) {
            Carry n[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) n[i] = carry(u + i);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                on = on && n[i].row == c.row;
                if (on) tot += n[i].val;
            }
            u += 8;
        }
        runs = __popc(__ballot_sync(0xffffffffu, on));
    }
    for (unsigned todo = __ballot_sync(0xffffffffu, on); todo; todo &= todo - 1) {
        const int src = __ffs(todo) - 1;
        const int row = __shfl_sync(0xffffffffu, c.row, src);
        double part = 0.0;
        bool more = true;
        for (int k = __shfl_sync(0xffffffffu, u, src) + lane; more; k += 256) {
            Carry n[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) n[i] = carry(k + 32 * i);
#pragma unroll
            for (int i = 0; i < 8; ++i)
                if (n[i].row == row) part += n[i].val;
            more = __all_sync(0xffffffffu, n[7].row == row);   // the run goes on past these 256
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) part += __shfl_xor_sync(0xffffffffu, part, off);
        if (lane == src) tot += part;
    }
    if (first) {
        const int o = a.rowmap ? __ldg(a.rowmap + c.row) : c.row;
        a.y[o] += tot;
    }
}

// Merge-path coordinates of every range boundary of a plan, computed on the
// device from a CSR row pointer: range t covers diagonals [t*ITEMS, (t+1)*ITEMS).
__global__ void merge_partition_kernel(const int32_t* __restrict__ ptr, int row_begin, int row_end,
                                       int32_t xoff, int per, MergeTile* __restrict__ tiles, int n_tiles) {
    const int t = (int)(blockIdx.x * blockDim.x + threadIdx.x);
    if (t >= n_tiles) return;
    const int k_base = __ldg(ptr + row_begin);
    const int a_len = row_end - row_begin;
    const int b_len = __ldg(ptr + row_end) - k_base;
    const int items = a_len + b_len;
    auto A = [&](int i) { return __ldg(ptr + row_begin + i + 1) - k_base; };
    const int d0 = t * per;
    const int d1 = d0 + per < items ? d0 + per : items;
    const int i0 = path_search(d0, a_len, b_len, A);
    const int i1 = path_search(d1, a_len, b_len, A);
    MergeTile m{};
    m.r0 = row_begin + i0;
    m.r1 = row_begin + i1;
    m.k0 = k_base + d0 - i0;
    m.k1 = k_base + d1 - i1;
    m.xoff = xoff;
    tiles[t] = m;
}

}  // namespace

int merge_plan_items(int64_t items) {
    return MERGE_CHUNK * (items <= 2 * (int64_t)MERGE_RANGES * MERGE_CHUNK ? 1 : 2) - MERGE_LANE;
}

// `items` (plan-free): merge items per range; else ranges [tile_begin, tile_end)
// of the plan's table.
template <bool PLAN>
static cudaError_t run_merge(const CsrArgs& a, const MergeTile* tiles, int tile_begin, int tile_end, int items,
                             Carry* carries, int num_sms, cudaStream_t s) {
    if (tile_end <= tile_begin) return cudaSuccess;
    const int n = tile_end - tile_begin;
    int grid = num_sms * 4;   // __launch_bounds__
    if (grid > (n + MERGE_WARPS - 1) / MERGE_WARPS) grid = (n + MERGE_WARPS - 1) / MERGE_WARPS;
    const bool a32 = PLAN || ((reinterpret_cast<uintptr_t>(a.col) | reinterpret_cast<uintptr_t>(a.val)) & 31) == 0;
    cudaError_t e = launch_pdl(a32 ? merge_kernel<PLAN, true> : merge_kernel<PLAN, PLAN>, dim3(grid), dim3(MERGE_NT), 0, s,
                               a, tiles, tile_begin, tile_end, items, carries);
    if (e != cudaSuccess) return e;
    return launch_pdl(merge_fixup_kernel, dim3((n + 255) / 256), dim3(256), 0, s, a, carries, tile_begin, tile_end);
}

cudaError_t launch_merge(const CsrArgs& a, const MergeTile* tiles, int tile_begin, int tile_end,
                         Carry* carries, int num_sms, cudaStream_t s) {
    return run_merge<true>(a, tiles, tile_begin, tile_end, 0, carries, num_sms, s);
}

int64_t merge_free_ranges(int64_t items) { return (items + range_items(items) - 1) / range_items(items); }

cudaError_t launch_merge_free(const CsrArgs& a, Carry* carries, int num_sms, cudaStream_t s) {
    const int64_t items = (int64_t)a.n_rows + a.nnz_total;
    return run_merge<false>(a, nullptr, 0, (int)merge_free_ranges(items), (int)range_items(items), carries, num_sms,
                            s);
}

cudaError_t launch_merge_partition(const int32_t* ptr, int row_begin, int row_end, int32_t xoff, int per,
                                   MergeTile* tiles, int n_tiles, cudaStream_t s) {
    if (n_tiles <= 0) return cudaSuccess;
    merge_partition_kernel<<<(n_tiles + 127) / 128, 128, 0, s>>>(ptr, row_begin, row_end, xoff, per, tiles,
                                                                 n_tiles);
    return cudaGetLastError();
}

cudaError_t read_clear_csr_error(int* out) {
    cudaError_t e = cudaMemcpyFromSymbol(out, g_csr_err, sizeof(int));
    if (e != cudaSuccess) return e;
    const int zero = 0;
    return cudaMemcpyToSymbol(g_csr_err, &zero, sizeof(int));
}

// ------------------------------------------------------------------------
// Fixed scratch for the no-allocation entry point.  Every GPU that loads the
// library holds this array until the process exits.  Its name is only a
// host-side stand-in in host code: the device address comes from
// cudaGetSymbolAddress, taken once per device with that device current.
// ------------------------------------------------------------------------
constexpr int64_t kNoAllocMaxItems = int64_t(65536) * 2048;   // the entry point's documented limit
static __device__ __align__(256) Carry g_noalloc_scratch[MERGE_RANGES];

namespace {
constexpr int kMaxDevices = 64;
std::mutex g_noalloc_mu;
void* g_noalloc_addr[kMaxDevices] = {};
}  // namespace

int64_t noalloc_max_items() { return kNoAllocMaxItems; }

cudaError_t launch_merge_noalloc(const CsrArgs& a, int num_sms, cudaStream_t s) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    void* base = nullptr;
    {
        std::lock_guard<std::mutex> lock(g_noalloc_mu);
        if (!g_noalloc_addr[dev]) {
            e = cudaGetSymbolAddress(&base, g_noalloc_scratch);
            if (e != cudaSuccess) return e;
            g_noalloc_addr[dev] = base;
        }
        base = g_noalloc_addr[dev];
    }
    const int64_t items = (int64_t)a.n_rows + a.nnz_total;
    if (items > noalloc_max_items()) return cudaErrorInvalidValue;
    // the carries of a launch are rewritten before they are read, so nothing
    // left by an earlier call is ever used
    return launch_merge_free(a, static_cast<Carry*>(base), num_sms, s);
}

}  // namespace spmvk
