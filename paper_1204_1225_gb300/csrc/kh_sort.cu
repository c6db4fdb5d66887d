// Binning sort of the traces (step before Eq. 1's sum): each trace gets its offset bin (the
// delta(X - |x_s - x_r|) of Eq. 1) and the cell of its midpoint on a coarse grid, and the
// traces are put in (bin, cell row, cell column, original index) order by a stable LSD radix
// sort over all SMs.  The (bin, cell) start table then lets a CTA of the migration walk only
// the cells that meet its tile's aperture disc (the traces near enough to carry the tile's
// reflections, Sec. 3 after Eq. 2) instead of its whole bin, so the staging work per CTA stays proportional to the
// traces it can use as surveys grow to tens of millions of traces (Sec. 2).
//
// Passes (each a few launches, no host synchronisation, no atomics on values, so the order is
// the same on every run):
//   k_cell_key      key = bin * ncell + cell, value = original index (dropped: key = nkeys)
//   k_radix_hist    per block of 4096 items, the counts of one 8-bit digit
//   k_radix_scan    exclusive scan of the counts, digit-major (one CTA)
//   k_radix_scatter stable scatter: items in index order, ranked per warp with match.any
//   k_key_starts    first sorted position of every key, and of every bin
// Up to SMALL_SORT traces everything after the keys (the passes, the starts, and the headers in sorted
// order) is one launch of one CTA, k_small_sort: the five or more launches are most of a short line's
// call, and their few blocks leave the chip idle either way.  (The keys stay a launch over all SMs:
// their FP64 offset takes 30 times a SM's share.)  Everything after the keys: 1024 traces 25 -> 6 us, 4608 traces 31 -> 9 us.
#include "kh_device.cuh"
#include "kh_plan.h"

namespace kh {

constexpr int RX_THREADS = 256;
constexpr int RX_ROUNDS = 16;
constexpr int RX_ITEMS = RX_THREADS * RX_ROUNDS;   // items per block
constexpr int RX_SCAN_THREADS = 1024;

int sort_hist_entries(int ntr) { return 256 * ((ntr + RX_ITEMS - 1) / RX_ITEMS); }

// Offset bin (FP64, as every kernel decides it) and midpoint cell (FP64 of the FP32 midpoint
// the aperture test uses).  Traces with no bin or a midpoint outside the grid get key nkeys.
__global__ void k_cell_key(int ntr, const float* __restrict__ sx, const float* __restrict__ sy,
                           const float* __restrict__ rx, const float* __restrict__ ry, int dim, int n_bins,
                           double w, CellGrid cg, int* __restrict__ key, int* __restrict__ val)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= ntr) return;
    const int ncell = cg.ncx * cg.ncy;
    const float a = sx[j], c = rx[j];
    const float b = (dim == 3 && sy) ? sy[j] : 0.f, d = (dim == 3 && ry) ? ry[j] : 0.f;
    const int bin = offset_bin(a, b, c, d, n_bins, w);
    int k = n_bins * ncell;
    if (bin >= 0) {
        int cx = 0, cy = 0;
        if (cg.margin > 0.0) {
            const float mx = __fmul_rn(__fadd_rn(a, c), 0.5f), my = __fmul_rn(__fadd_rn(b, d), 0.5f);
            const double fx = floor(__dmul_rn(__dadd_rn((double)mx, -cg.gx0), cg.inv_cs));
            const double fy = (dim == 3) ? floor(__dmul_rn(__dadd_rn((double)my, -cg.gy0), cg.inv_cs)) : 0.0;
            const bool in_grid = fx >= 0.0 && fx < (double)cg.ncx && fy >= 0.0 && fy < (double)cg.ncy;
            if (in_grid) {
                cx = (int)fx;
                cy = (int)fy;
                k = bin * ncell + cy * cg.ncx + cx;
            }
        } else {
            k = bin * ncell;
        }
    }
    key[j] = k;
    val[j] = j;
}

__global__ void __launch_bounds__(RX_THREADS) k_radix_hist(int n, const int* __restrict__ key, int shift,
                                                           int* __restrict__ hist, int nblocks)
{
    __shared__ int cnt[256];
    const int tid = threadIdx.x;
    cnt[tid] = 0;
    __syncthreads();
    const int base = blockIdx.x * RX_ITEMS;
    for (int r = 0; r < RX_ROUNDS; ++r) {
        const int i = base + r * RX_THREADS + tid;
        if (i < n) atomicAdd(&cnt[(key[i] >> shift) & 255], 1);
    }
    __syncthreads();
    hist[tid * nblocks + blockIdx.x] = cnt[tid];
}

// Exclusive scan of `n` counts in place, one CTA: each thread sums a contiguous chunk, the
// chunk sums are scanned in shared memory, then each thread rewrites its chunk.
__global__ void __launch_bounds__(RX_SCAN_THREADS) k_radix_scan(int* __restrict__ a, int n)
{
    __shared__ int part[RX_SCAN_THREADS];
    const int tid = threadIdx.x;
    const int chunk = (n + RX_SCAN_THREADS - 1) / RX_SCAN_THREADS;
    const int lo = min(n, tid * chunk), hi = min(n, lo + chunk);
    int sum = 0;
    for (int i = lo; i < hi; ++i) sum += a[i];
    part[tid] = sum;
    __syncthreads();
    for (int o = 1; o < RX_SCAN_THREADS; o <<= 1) {   // Hillis-Steele inclusive scan
        const int v = tid >= o ? part[tid - o] : 0;
        __syncthreads();
        part[tid] += v;
        __syncthreads();
    }
    int run = part[tid] - sum;
    for (int i = lo; i < hi; ++i) {
        const int c = a[i];
        a[i] = run;
        run += c;
    }
}

// Stable scatter of one digit: the block's items in index order, 256 per round; within a warp
// the items of equal digit are ranked by lane (match.any), across warps by warp order.
__global__ void __launch_bounds__(RX_THREADS)
    k_radix_scatter(int n, const int* __restrict__ kin, const int* __restrict__ vin, int* __restrict__ kout,
                    int* __restrict__ vout, int shift, const int* __restrict__ offs, int nblocks)
{
    constexpr int WARPS = RX_THREADS / 32;
    __shared__ int base[256];
    __shared__ int wcnt[WARPS][256];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    base[tid] = offs[tid * nblocks + blockIdx.x];
    const unsigned lt = (1u << lane) - 1u;
    for (int r = 0; r < RX_ROUNDS; ++r) {
        const int i = blockIdx.x * RX_ITEMS + r * RX_THREADS + tid;
#pragma unroll
        for (int w = 0; w < WARPS; ++w) wcnt[w][tid] = 0;
        __syncthreads();
        const bool valid = i < n;
        const int k = valid ? kin[i] : 0;
        const int d = valid ? (k >> shift) & 255 : 256;
        const unsigned same = __match_any_sync(0xffffffffu, d);
        const int rank = __popc(same & lt);
        if (valid && rank == 0) wcnt[warp][d] = __popc(same);
        __syncthreads();
        int run = 0;
#pragma unroll
        for (int w = 0; w < WARPS; ++w) {
            const int c = wcnt[w][tid];
            wcnt[w][tid] = run;
            run += c;
        }
        __syncthreads();
        if (valid) {
            const int pos = base[d] + wcnt[warp][d] + rank;
            kout[pos] = k;
            vout[pos] = vin[i];
        }
        __syncthreads();
        base[tid] += run;
    }
}

// start[k] = first sorted position whose key is >= k, for k = 0 .. nkeys (start[nkeys] = number
// of kept traces); bin_start[b] = start[b * ncell].
__global__ void k_key_starts(int n, const int* __restrict__ key, int nkeys, int ncell, int* __restrict__ start,
                             int* __restrict__ bin_start)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i <= n; i += gridDim.x * blockDim.x) {
        const int prev = i == 0 ? -1 : min(key[i - 1], nkeys);
        const int cur = i == n ? nkeys : min(key[i], nkeys);
        for (int k = prev + 1; k <= cur; ++k) {
            start[k] = i;
            if (k % ncell == 0) bin_start[k / ncell] = i;
        }
    }
}

constexpr int SMALL_SORT = 8192;   // 16-bit indexes; keys, values and counts fit one CTA's shared memory
constexpr int SS_THREADS = 1024, SS_WARPS = SS_THREADS / 32;

struct SmallSortSmem {
    int key[2][SMALL_SORT];
    unsigned short val[2][SMALL_SORT];
    int cnt[SS_WARPS][256];   // a warp's next position of each digit
    int total[256];
};

// Stable LSD radix sort in shared memory: each warp owns a contiguous chunk of the items and walks it in
// order, 32 at a time, ranked by match.any; counts are scanned digit-major, then warp.
__global__ void __launch_bounds__(SS_THREADS)
    k_small_sort(int n, const int* __restrict__ key_in, int passes, int nkeys, int ncell,
                 const float* __restrict__ sx, const float* __restrict__ sy, const float* __restrict__ rx,
                 const float* __restrict__ ry, int dim, int* __restrict__ perm, int* __restrict__ start,
                 int* __restrict__ bin_start, float4* __restrict__ hdr, float2* __restrict__ mid)
{
    extern __shared__ __align__(16) unsigned char ss_smem[];
    SmallSortSmem& S = *reinterpret_cast<SmallSortSmem*>(ss_smem);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int i = tid; i < n; i += SS_THREADS) {
        S.key[0][i] = key_in[i];
        S.val[0][i] = (unsigned short)i;
    }
    const int chunk = (n + SS_THREADS - 1) / SS_THREADS * 32;   // items of a warp
    const int first = min(n, warp * chunk), last = min(n, first + chunk);
    const unsigned lt = (1u << lane) - 1u;
    int cur = 0;
    for (int p = 0; p < passes; ++p, cur ^= 1) {
        const int shift = 8 * p;
        for (int d = lane; d < 256; d += 32) S.cnt[warp][d] = 0;
        __syncthreads();
        for (int i = first + lane; i - lane < last; i += 32) {
            const int d = i < last ? (S.key[cur][i] >> shift) & 255 : 256;
            const unsigned same = __match_any_sync(0xffffffffu, d);
            if (d < 256 && (same & lt) == 0) S.cnt[warp][d] += __popc(same);
            __syncwarp();
        }
        __syncthreads();
        if (tid < 256) {
            int run = 0;
            for (int w = 0; w < SS_WARPS; ++w) {
                const int c = S.cnt[w][tid];
                S.cnt[w][tid] = run;
                run += c;
            }
            S.total[tid] = run;
        }
        __syncthreads();
        if (warp == 0) {   // exclusive scan of the 256 totals, eight a lane
            int v[8], sum = 0;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                v[k] = sum;
                sum += S.total[lane * 8 + k];
            }
            int pre = sum;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, pre, o);
                if (lane >= o) pre += u;
            }
#pragma unroll
            for (int k = 0; k < 8; ++k) S.total[lane * 8 + k] = pre - sum + v[k];
        }
        __syncthreads();
        for (int i = first + lane; i - lane < last; i += 32) {
            const int k = i < last ? S.key[cur][i] : 0;
            const int d = i < last ? (k >> shift) & 255 : 256;
            const unsigned same = __match_any_sync(0xffffffffu, d);
            const int rank = __popc(same & lt);
            int pos = 0;
            if (d < 256) pos = S.total[d] + S.cnt[warp][d] + rank;
            __syncwarp();
            if (d < 256) {
                if (rank == 0) S.cnt[warp][d] += __popc(same);
                S.key[cur ^ 1][pos] = k;
                S.val[cur ^ 1][pos] = S.val[cur][i];
            }
            __syncwarp();
        }
        __syncthreads();
    }
    for (int i = tid; i <= n; i += SS_THREADS) {   // as k_key_starts
        const int prev = i == 0 ? -1 : min(S.key[cur][i - 1], nkeys);
        const int k1 = i == n ? nkeys : min(S.key[cur][i], nkeys);
        for (int k = prev + 1; k <= k1; ++k) {
            start[k] = i;
            if (k % ncell == 0) bin_start[k / ncell] = i;
        }
        if (i == n) continue;
        const int j = S.val[cur][i];
        perm[i] = j;
        if (S.key[cur][i] >= nkeys) continue;   // dropped: no header is read
        const float a = sx[j], c = rx[j];
        const float b = (dim == 3 && sy) ? sy[j] : 0.f, d = (dim == 3 && ry) ? ry[j] : 0.f;
        hdr[i] = make_float4(a, b, c, d);
        mid[i] = make_float2(__fmul_rn(__fadd_rn(a, c), 0.5f), __fmul_rn(__fadd_rn(b, d), 0.5f));
    }
}

bool sorts_in_one(int ntr) { return ntr <= SMALL_SORT; }

cudaError_t sort_traces(int ntr, const float* sx, const float* sy, const float* rx, const float* ry,
                        int dim, int n_bins, double bin_width, const CellGrid& cg, int* key_a,
                        int* key_b, int* val_a, int* val_b, int* hist, int* cell_start, int* bin_start,
                        float4* hdr, float2* mid, const int** perm_out, int* launches, cudaStream_t s)
{
    const int ncell = cg.ncx * cg.ncy;
    const int nkeys = n_bins * ncell;
    int bits = 1;
    while ((1LL << bits) <= (long long)nkeys) ++bits;   // keys are 0 .. nkeys
    const int passes = (bits + 7) / 8;
    const int nblocks = (ntr + RX_ITEMS - 1) / RX_ITEMS;
    int *kin = key_a, *kout = key_b, *vin = val_a, *vout = val_b;
    if (ntr > 0) {
        k_cell_key<<<(ntr + 255) / 256, 256, 0, s>>>(ntr, sx, sy, rx, ry, dim, n_bins, bin_width, cg, kin, vin);
        ++*launches;
        if (sorts_in_one(ntr)) {
            const cudaError_t e = cudaFuncSetAttribute(k_small_sort, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                       (int)sizeof(SmallSortSmem));
            if (e != cudaSuccess) return e;
            k_small_sort<<<1, SS_THREADS, sizeof(SmallSortSmem), s>>>(ntr, kin, passes, nkeys, ncell, sx, sy, rx, ry,
                                                                       dim, vin, cell_start, bin_start, hdr, mid);
            ++*launches;
            *perm_out = vin;
            return cudaGetLastError();
        }
        for (int p = 0; p < passes; ++p) {
            k_radix_hist<<<nblocks, RX_THREADS, 0, s>>>(ntr, kin, 8 * p, hist, nblocks);
            k_radix_scan<<<1, RX_SCAN_THREADS, 0, s>>>(hist, 256 * nblocks);
            k_radix_scatter<<<nblocks, RX_THREADS, 0, s>>>(ntr, kin, vin, kout, vout, 8 * p, hist, nblocks);
            *launches += 3;
            int* t = kin;
            kin = kout;
            kout = t;
            t = vin;
            vin = vout;
            vout = t;
        }
    }
    const int blocks = std::max(1, std::min((ntr + 256) / 256, 4096));
    k_key_starts<<<blocks, 256, 0, s>>>(ntr, kin, nkeys, ncell, cell_start, bin_start);
    *launches += 2;
    *perm_out = vin;
    return launch_gather(ntr, bin_start, n_bins, vin, sx, sy, rx, ry, dim, hdr, mid, s);
}

}  // namespace kh
