// Migration kernel (Eq. 1, Sec. 3): output-stationary gather over an image tile and one
// offset bin.
//
// CTA = 8 consumer warps + 1 producer warp.  Each consumer thread owns NZ = 16 consecutive
// z samples of one image column and keeps their FP32 accumulators in registers for the
// whole kernel; nothing is accumulated in global memory.  The producer warp walks the
// bin's traces (sorted by bin), culls those whose midpoint is outside the aperture of the
// tile footprint, bounds the two-way time over the tile box to a sample window
// [lo, hi], computes the trace's FP64 reference at the tile centre (linear v(z)), and
// stages the window into a 3-deep shared-memory ring with one cp.async.bulk per trace
// (16-byte aligned, no multicast) completing on the stage's mbarrier.  Traces arrive
// as FP32 (sample, step) pairs, so one 8-byte shared load and one FMA give an interpolated sample
// (plain samples where a pair row does not fit, see use_pairs).
// Consumers evaluate tau for their points (kh_tau.cuh; linear v(z): per-leg logarithms with the
// source leg cached per source position), read the staged samples, interpolate linearly,
// weight and accumulate; a warp whose window is not clipped and whose lanes all lie in the
// aperture and the grid skips the validity test.  All mbarrier waits are bounded; a wait that
// runs out sets the plan's status word and the CTA leaves only after its copies have landed.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <cstddef>
#include <type_traits>

#include "kh_f32x2.cuh"
#include "kh_tau.cuh"

namespace kh {

template <typename TT>
__device__ __forceinline__ float to_f32(TT v);
template <>
__device__ __forceinline__ float to_f32<float>(float v) { return v; }
template <>
__device__ __forceinline__ float to_f32<__half>(__half v) { return __half2float(v); }
template <>
__device__ __forceinline__ float to_f32<__nv_bfloat16>(__nv_bfloat16 v) { return __bfloat162float(v); }

constexpr int MAX_ZG = 16;          // z-groups per CTA (cz)
constexpr int SLACK = 16;           // zeroed elements after the ring (reads one past a window)
constexpr int LEAD = 16;            // zeroed elements before the ring (a window clipped at t0 may be
                                    // indexed at -1 when tau is a rounding error below 0)

struct __align__(16) MigSmem {
    uint64_t full[STAGES];
    uint64_t empty[STAGES];
    int cnt[STAGES];
    int last[STAGES];
    int row[4];                 // cell range of the tile (cx0, cx1, first row - 1, last row)
    int2 rng[MAX_CELL_ROWS];    // staging warp: sorted trace range of each cell row of the tile
    unsigned stat[2];           // staging warp: traces examined and staged for this tile
    // per staged trace
    float4 hdr[STAGES][BMAX];   // (sx, sy, rx, ry)
    float4 hda[STAGES][BMAX];   // linear: (c_x-2s_x, c_y-2s_y, c_x-2r_x, c_y-2r_y)
    float4 refs[STAGES][BMAX];  // linear: source-leg LegRef
    float4 refr[STAGES][BMAX];  // linear: receiver-leg LegRef
    float2 mid[STAGES][BMAX];   // FP32 midpoint (aperture test)
    int4 win[STAGES][BMAX];     // x: tau_ref - lo (float bits), y: smem index of sample lo minus
                                // MAGIC_BITS, z/w: c_mid/c_half (float bits) of the valid range
                                // 0 <= tau - lo <= hi - lo (EDGE_EPS wider on each side); sign
                                // bit of z: every column of the
                                // tile inside the aperture; sign bit of w: window not clipped
    float tb[STAGES][BMAX];     // lo dt + t0: T_s + T_r = (tau - lo) dt + tb (gradient mode)
    float4 zc[MAX_ZG * NZ];     // per-z constants (tile_z_setup)
    float z2[MAX_ZG * NZ];      // depth factor of the weight (linear: gamma(z))
    float zero[4];
};
static_assert(offsetof(MigSmem, zero) % 16 == 0, "the zero sample (pair) must be 16-byte aligned");

__host__ __device__ constexpr size_t mig_static_bytes() { return (sizeof(MigSmem) + 127) / 128 * 128; }

// Dynamic shared memory of one CTA when two CTAs share an SM's 228 KB (the runtime reserves
// 1 KB per CTA; 128 B of static shared variables).
constexpr size_t CTA_SMEM_BUDGET = 228 * 1024 / 2 - 1024 - 128;

// Nodes [tnh][tnz] (16-byte padded), then for KH_F16 one float4 (c0, c1, c2, 0) per h row: the
// row's reference polynomial in the normalised node depth (the nodes hold T minus it in FP16).
__host__ __device__ inline size_t table_node_bytes(const GeomParams& g)
{
    const size_t es = g.tdt == KH_F32 ? 4 : 2;
    return ((size_t)g.tnh * g.tnz * es + 15) / 16 * 16;
}

__host__ __device__ inline size_t table_bytes(const GeomParams& g)
{
    if (!g.table) return 0;
    return table_node_bytes(g) + (g.tdt == KH_F16 ? (size_t)g.tnh * sizeof(float4) : 0);
}

// Per consumer thread and depth, the cached source leg of the current source position (see
// mig_consumer): (C1 ln(1 + rho_s), sqrt(q_s)) for linear v(z), (dR_s, R_s) for time migration,
// (dR_s, 1/R_s) for the constant-velocity true-amplitude kernels, T_s for the tables (the radial table's shared copy
// leaves no room for more at two CTAs per SM).  The other constant-velocity kernels keep no cache:
// their leg is one square root, and surveys whose traces do not arrive shot by shot (the batched
// jobs') would recompute it per trace anyway.
__host__ __device__ inline size_t src_cache_bytes(const GeomParams& g)
{
    if (g.table || g.gtab) return (size_t)NZ * CONSUMERS * sizeof(float);
    // gradient: the thread's weighted image values, and for linear v(z) (C1 ln(1 + rho_s), (q/w)_s)
    // and sqrt(q_s)
    if (g.grad) return (size_t)NZ * CONSUMERS * (g.kabs > 0.0 ? sizeof(float2) + 2 * sizeof(float) : sizeof(float));
    return (g.kabs > 0.0 || g.pstm || g.weight == KH_W_TRUE_AMP) ? (size_t)NZ * CONSUMERS * sizeof(float2) : 0;
}

// Elements of one stage's sample area: a full trace always fits, so every trace is stageable (with a
// traveltime table and pairs, the longest window any tile can ask for: win_max).
// Plain samples: 16 KB per stage.  SamplePair rows hold half as many samples per byte; they take
// the largest stage at which two CTAs of the linear path (static part, ring, 32 KB source-leg
// cache) still fit.  With a traveltime table, the largest stage up to 16 KB at which two CTAs
// fit beside the table, but at least 8 KB (a large F32 table then runs one CTA per SM).  The
// gradient kernel's 64 KB of per-thread data leaves 8.75 KB per stage of slope rows at two CTAs
// per SM.
constexpr int PAIR_STAGE_BYTES = 19712;   // 2464 pairs, 1 KB of margin per SM
static_assert(((sizeof(MigSmem) + 127) / 128 * 128) +
                      ((LEAD + STAGES * (PAIR_STAGE_BYTES / 8) + SLACK) * 8 + 15) / 16 * 16 +
                      NZ * CONSUMERS * sizeof(float2) <= CTA_SMEM_BUDGET,
              "two CTAs of the pair-staged linear kernel must fit on one SM");
static_assert(PAIR_STAGE_BYTES / 8 >= (PAIR_MAX_NT + 5) / 2 * 2, "a whole pair row must fit one stage");
static_assert(((sizeof(MigSmem) + 127) / 128 * 128) + ((LEAD + STAGES * (8960 / 4) + SLACK) * 4 + 15) / 16 * 16 +
                      NZ * CONSUMERS * (sizeof(float2) + 2 * sizeof(float)) <= CTA_SMEM_BUDGET,
              "two CTAs of the linear gradient kernel must fit on one SM");
__host__ __device__ inline int mig_cap(const GeomParams& g)
{
    const int ealign = g.elem_align;
    const int need = ((g.win_max ? g.win_max : g.nt) + 2 * ealign + ealign - 1) / ealign * ealign;
    long long bytes = g.grad ? 8960 : g.pairs ? PAIR_STAGE_BYTES : 16384;
    if (g.table) {
        const long long room = (long long)CTA_SMEM_BUDGET - (long long)mig_static_bytes() -
                               (long long)table_bytes(g) - (long long)src_cache_bytes(g) -
                               (long long)(LEAD + SLACK) * g.esize - 16;
        bytes = room / STAGES / 1024 * 1024;
        bytes = bytes > 16384 ? 16384 : (bytes < 8192 ? 8192 : bytes);
    }
    const int base = (int)(bytes / g.esize);
    return need > base ? need : base;
}

__host__ __device__ inline size_t mig_ring_bytes(const GeomParams& g)
{
    return (((size_t)LEAD + STAGES * mig_cap(g) + SLACK) * g.esize + 15) / 16 * 16;
}

inline size_t mig_smem_bytes(const GeomParams& g)
{
    return mig_static_bytes() + mig_ring_bytes(g) + table_bytes(g) + src_cache_bytes(g);
}

// Radial table, step 1 (once per thread and trace leg): the table interpolated in h at the
// horizontal distance sqrt(dh2), at the K depth nodes jb .. jb + K - 1 that span the thread's
// 16 depths.
template <typename TB, int K, bool FAST>
__device__ __forceinline__ void tab_profile(const TB* tab, const GeomParams& g, float dh2, int jb, float* p)
{
    const float u = fminf(hsqrt<FAST>(dh2) * g.tinv, g.thmax);
    const int ih = (int)u;
    const float fh = u - (float)ih;
    // two nodes a load: rows and first nodes are even (16 / M nodes a thread, two to spare a row), and the
    // load of the last, odd node reads its row's spare one too
    const TB* r0 = tab + ih * g.tnz + jb;
    const TB* r1 = r0 + g.tnz;
    const F2 fh2 = f2(fh);
#pragma unroll
    for (int k = 0; k < K; k += 2) {
        F2 a, d;
        if constexpr (sizeof(TB) == 4) {
            a = *reinterpret_cast<const F2*>(r0 + k);
            d = sub2(*reinterpret_cast<const F2*>(r1 + k), a);
        } else {
            const unsigned wa = *reinterpret_cast<const unsigned*>(r0 + k), wb = *reinterpret_cast<const unsigned*>(r1 + k);
            if constexpr (std::is_same<TB, __half>::value) {
                const float2 fa = __half22float2(*reinterpret_cast<const __half2*>(&wa));
                const float2 fb = __half22float2(*reinterpret_cast<const __half2*>(&wb));
                a = f2(fa.x, fa.y);
                d = sub2(f2(fb.x, fb.y), a);
            } else {   // 2^23 + u has u in its low mantissa bits
                const F2 ua = f2(__uint_as_float(__byte_perm(wa, 0x4B000000u, 0x7410)), __uint_as_float(__byte_perm(wa, 0x4B000000u, 0x7432)));
                const F2 ub = f2(__uint_as_float(__byte_perm(wb, 0x4B000000u, 0x7410)), __uint_as_float(__byte_perm(wb, 0x4B000000u, 0x7432)));
                d = sub2(ub, ua);
                a = sub2(ua, f2(8388608.f));
            }
        }
        const float2 v = f2_get(fma2(fh2, d, a));
        p[k] = v.x;
        if (k + 1 < K) p[k + 1] = v.y;
    }
    if constexpr (std::is_same<TB, __half>::value) {
        // FP16 residuals: add the rows' reference polynomials, interpolated in h like the nodes
        // (the interpolation is linear in the coefficients)
        const float4* cf = reinterpret_cast<const float4*>(reinterpret_cast<const char*>(tab) + table_node_bytes(g));
        const float4 q0 = cf[ih], q1 = cf[ih + 1];
        const float c0 = fmaf(fh, q1.x - q0.x, q0.x), c1 = fmaf(fh, q1.y - q0.y, q0.y);
        const float c2 = fmaf(fh, q1.z - q0.z, q0.z);
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const float u = (float)(jb + k) * g.tunz;
            p[k] += fmaf(fmaf(c2, u, c1), u, c0);
        }
    }
}

// Step 2 (per depth): depth nodes sit every M image samples from the thread's first depth,
// so depth i lies in node interval i / M at fraction (i % M) / M, both compile-time.
template <int M>
__device__ __forceinline__ float tab_depth(const float* p, int i)
{
    const int j = i / M, r = i % M;
    return r == 0 ? p[j] : fmaf((float)r * (1.f / M), p[j + 1] - p[j], p[j]);
}

// One leg's profile at K node rows from its location's table ([row][column], x fastest): the lerp
// in x between the column's two node columns (c0 points at node column gi of the first row; the
// next row follows gnx later).  The lanes of a warp (consecutive image columns) read a few
// consecutive nodes of one row per load.
template <int K>
__device__ __forceinline__ void grid_profile(const float* __restrict__ c0, int gnx, float fx, float* p)
{
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const float a = __ldg(c0 + k * gnx), b = __ldg(c0 + k * gnx + 1);
        p[k] = fmaf(fx, b - a, a);
    }
}

// The migration kernel's sample reads, two depths at a time: th = tau - lo (window-relative
// sample position); linear interpolation between samples floor(th) and floor(th) + 1 (adding
// 1.5 * 2^23 rounded down leaves floor(th) in the low mantissa bits).
template <typename TT>
__device__ __forceinline__ float lerp_at(const TT* data, int off, float f)
{
    if constexpr (std::is_same<TT, SamplePair>::value) {
        const float2 p = *reinterpret_cast<const float2*>(data + off);
        return fmaf(f, p.y, p.x);
    } else {
        const float d0 = to_f32<TT>(data[off]);
        const float d1 = to_f32<TT>(data[off + 1]);
        return fmaf(f, d1 - d0, d0);
    }
}

// Valid iff |th - cmid| <= chalf, i.e. 0 <= th <= hi - lo up to EDGE_EPS; th below 0 read as 0;
// invalid points read the zeros at zero_off.
template <typename TT>
__device__ __forceinline__ F2 sample2_at(const TT* data, F2 th2, int base, float cmid, float chalf, int zero_off)
{
    const float2 t = f2_get(th2);
    const bool ok0 = fabsf(t.x - cmid) <= chalf, ok1 = fabsf(t.y - cmid) <= chalf;
    const F2 tc = f2(fmaxf(t.x, 0.f), fmaxf(t.y, 0.f));
    const F2 tm2 = add2_rd(tc, f2(MAGIC));
    const float2 f = f2_get(sub2(tc, sub2(tm2, f2(MAGIC))));
    const float2 tm = f2_get(tm2);
    return f2(lerp_at<TT>(data, ok0 ? __float_as_int(tm.x) + base : zero_off, f.x),
              lerp_at<TT>(data, ok1 ? __float_as_int(tm.y) + base : zero_off, f.y));
}

// sample2_at without the validity test, for traces whose window is not clipped and whose every
// lane and depth lies in the tile box (so 0 <= th <= hi - lo).  Indexes the ring from its
// lead (base + LEAD); the unsigned clamp to the last readable pair keeps any index in bounds.
template <typename TT>
__device__ __forceinline__ F2 sample2_unchecked(const TT* ring, F2 th2, int base_lead, unsigned last)
{
    const F2 tm2 = add2_rd(th2, f2(MAGIC));
    const float2 f = f2_get(sub2(th2, sub2(tm2, f2(MAGIC))));
    const float2 tm = f2_get(tm2);
    return f2(lerp_at<TT>(ring, (int)min((unsigned)(__float_as_int(tm.x) + base_lead), last), f.x),
              lerp_at<TT>(ring, (int)min((unsigned)(__float_as_int(tm.y) + base_lead), last), f.y));
}

// ------------------------------------------------------------------ producer warp
// The sorted traces one CTA examines: its bin's whole range, or with a (bin, cell) start table
// one range per row of the cells that meet the tile footprint widened by the aperture margin
// (cells of a row are consecutive in the sort order).  Every trace the staging cull would keep
// lies in those cells: its midpoint is within the cull radius, margin - 1 m, of the footprint.
// The row state (cx0, cx1, current row, last row) lives in shared memory, written by the
// staging warp only: it changes once per cell row, and keeping it out of registers leaves the
// kernel's register budget to the consumers.
// The tile's cell range, written by one thread before the tile's set-up barrier.
__device__ __forceinline__ void tile_cells(int* row, const TraceSet& tr, const TileBox& box)
{
    if (!tr.cell_start) return;
    const CellGrid& cg = tr.cg;
    auto cell = [&](double v, double g0, int n) {
        const double f = floor((v - g0) * cg.inv_cs);
        return (int)fmin(fmax(f, -1.0), (double)n);
    };
    const int cx0 = max(0, cell((double)box.xlo - cg.margin, cg.gx0, cg.ncx));
    const int cx1 = min(cg.ncx - 1, cell((double)box.xhi + cg.margin, cg.gx0, cg.ncx));
    const int cy0 = max(0, cell((double)box.ylo - cg.margin, cg.gy0, cg.ncy));
    const int cy1 = min(cg.ncy - 1, cell((double)box.yhi + cg.margin, cg.gy0, cg.ncy));
    row[0] = cx0;
    row[1] = cx1;
    row[2] = cy0 - 1;
    row[3] = (cx0 <= cx1) ? cy1 : cy0 - 1;
}

// Part `split` of `n` of a sorted trace range that starts at position `pre` of the tile's `total`:
// the parts are consecutive, their lengths a trace apart.
__device__ __forceinline__ int2 cut_range(int2 r, int pre, int total, int split, int n)
{
    if (n == 1) return r;
    const int len = r.y - r.x;
    const int lo = (int)((long long)total * split / n) - pre, hi = (int)((long long)total * (split + 1) / n) - pre;
    return make_int2(r.x + min(max(lo, 0), len), r.x + min(max(hi, 0), len));
}

// The tile's sorted trace range of every cell row (its part of them, see cut_range), written by the
// staging warp into shared memory (rng[0 .. nr - 1]); the walk keeps its row index and count in
// shared memory too (row[2], row[3]), so that it adds no register to the staging loop.
__device__ __forceinline__ void tile_rows(int* row, int2* rng, const TraceSet& tr, int bin, int split, int nsplit)
{
    static_assert(MAX_CELL_ROWS <= 32, "a lane per cell row");
    const int ncx = tr.cg.ncx;
    const int* cs = tr.cell_start + (long long)bin * ncx * tr.cg.ncy;
    const int cx0 = row[0], cx1 = row[1], cy0 = row[2] + 1, nr = row[3] - row[2];
    const int i = threadIdx.x & 31;
    int2 r = make_int2(0, 0);
    if (i < nr) r = make_int2(cs[(cy0 + i) * ncx + cx0], cs[(cy0 + i) * ncx + cx1 + 1]);
    int pre = r.y - r.x;   // inclusive prefix of the rows' lengths
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, pre, o);
        if (i >= o) pre += v;
    }
    const int total = __shfl_sync(0xffffffffu, pre, 31);
    if (i < nr) rng[i] = cut_range(r, pre - (r.y - r.x), total, split, nsplit);
    __syncwarp();
    if ((threadIdx.x & 31) == 0) {
        row[2] = -1;
        row[3] = nr;
    }
    __syncwarp();
}

// Moves (cur, te) to the next non-empty cell row; leaves cur >= te when none is left.
__device__ __forceinline__ void next_row(int* row, const int2* rng, int& cur, int& te)
{
    int ri = row[2];
    const int nr = row[3];
    while (cur >= te && ri + 1 < nr) {
        ++ri;
        cur = rng[ri].x;
        te = rng[ri].y;
    }
    __syncwarp();
    if ((threadIdx.x & 31) == 0) row[2] = ri;
    __syncwarp();
}

// `n` is the number of stages this CTA's producer has filled before (mbarrier phases carry
// over from one work item to the next in the persistent kernel); returns the new count.
// The window-relative time the consumers evaluate is tau - lo (sample index floor(tau - lo)).
template <int VEL, typename TT, int WGT = 0>
__device__ __forceinline__ int mig_producer(MigSmem& S, TT* data, int cap, const GeomParams& g,
                                            const TraceSet& tr, const TT* __restrict__ traces, int bin,
                                            const TileBox& box, const WaitCfg& wc, int n, int tile_id, int split,
                                            int nsplit)
{
    const int lane = threadIdx.x & 31;
    const double inv_kdt = (VEL == VK_LINEAR) ? 1.0 / (g.kabs * g.dtd) : 0.0;
    PstmTile pt{};
    if constexpr (VEL == VK_PSTM) pt = pstm_tile(g, box);
    int cur = tr.bin_start[bin], te = tr.bin_start[bin + 1];
    const int2 part = cut_range(make_int2(cur, te), 0, te - cur, split, nsplit);
    cur = part.x;
    te = part.y;
    if (tr.cell_start) {   // the first non-empty cell row of the tile
        tile_rows(S.row, S.rng, tr, bin, split, nsplit);
        cur = te = 0;
        next_row(S.row, S.rng, cur, te);
    }
    if (lane == 0) S.stat[0] = S.stat[1] = 0u;
    const int n_begin = n;
    bool failed = false;
    while (true) {
        const int s = n % STAGES;
        if (n >= STAGES) {
            if (!warp_wait(&S.empty[s], ((n / STAGES) - 1) & 1, wc.polls, wc.ns, wc.status)) {
                failed = true;
                break;
            }
        }
        int cnt = 0, used = 0;
        bool full = false;
        while (cur < te && !full) {
            const int k = cur + lane;
            bool ok = false;
            int lo = 0, hi = 0, lo_al = 0, len_al = 0;
            bool clipped = true;
            float4 h = make_float4(0.f, 0.f, 0.f, 0.f);
            float2 m = make_float2(0.f, 0.f);
            if (k < te) {
                h = tr.hdr[k];
                m = tr.mid[k];
                ok = true;
                if (g.use_aperture) {
                    const float ax = fmaxf(fmaxf(box.xlo - m.x, m.x - box.xhi), 0.f);
                    const float ay = fmaxf(fmaxf(box.ylo - m.y, m.y - box.yhi), 0.f);
                    ok = ax * ax + ay * ay <= g.A2cull;
                }
                if (ok) {
                    if constexpr (VEL == VK_GRID) {
                        // the window from the tile's node bounds of both legs' tables; a negative
                        // location (a position with no table) skips the trace
                        const int ls = __float_as_int(h.y), lr = __float_as_int(h.w);
                        ok = ls >= 0 && lr >= 0;
                        if (ok) {
                            const float2 bs = __ldg(&g.gbnd[(long long)ls * g.gtiles + tile_id]);
                            const float2 br = __ldg(&g.gbnd[(long long)lr * g.gtiles + tile_id]);
                            ok = sample_window(__fadd_rn(bs.x, br.x), __fadd_rn(bs.y, br.y), g, lo, hi, &clipped);
                        }
                    } else {
                        ok = trace_window(h, box, VEL == VK_TABLE ? (g.k == 0.0 ? VK_CONST : VK_LINEAR) : VEL,
                                          g, lo, hi, &clipped, &pt);
                    }
                    lo_al = lo & ~(g.elem_align - 1);
                    len_al = (hi + 1 - lo_al + g.elem_align - 1) & ~(g.elem_align - 1);
                    if (ok && len_al > cap) {   // the host's bound excludes it; an unstageable window would never end
                        atomicOr(wc.status, 2);
                        ok = false;
                    }
                }
            }
            const unsigned okm = __ballot_sync(0xffffffffu, ok);
            int pre = ok ? len_al : 0;   // inclusive prefix of window lengths
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, pre, o);
                if (lane >= o) pre += v;
            }
            const int excl = pre - (ok ? len_al : 0);
            const int rank = __popc(okm & ((1u << lane) - 1u));
            const bool fits = ok && (cnt + rank < BMAX) && (used + excl + len_al <= cap);
            const unsigned fm = __ballot_sync(0xffffffffu, fits);
            const unsigned nofit = okm & ~fm;
            const int consumed = nofit ? (__ffs(nofit) - 1) : min(32, te - cur);
            const int nfit = __popc(fm);
            int bytes = fits ? len_al * g.esize : 0;
            int used_add = fits ? len_al : 0;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                bytes += __shfl_xor_sync(0xffffffffu, bytes, o);
                used_add += __shfl_xor_sync(0xffffffffu, used_add, o);
            }
            if (fits) {
                const int slot = cnt + rank;
                const int dst = s * cap + used + excl;
                double tau_ref = (VEL == VK_TABLE) ? g.c0 + 0.5 : -g.t0d / g.dtd;
                if constexpr (VEL == VK_LINEAR) {
                    LegRef rs, rr;
                    float qis = 0.f, qir = 0.f;
                    const double ls = leg_reference(box.cx, box.cy, box.cz, h.x, h.y, g, rs, &qis);
                    const double lr = leg_reference(box.cx, box.cy, box.cz, h.z, h.w, g, rr, &qir);
                    tau_ref = __dadd_rn(tau_ref, __dmul_rn(__dadd_rn(ls, lr), inv_kdt));
                    // (R_c^2, (q_c + 2)/u_c, w_c, 1/u_c) per leg
                    S.refs[s][slot] = make_float4(rs.Rc2, qis, rs.wc, rs.iuc);
                    S.refr[s][slot] = make_float4(rr.Rc2, qir, rr.wc, rr.iuc);
                    S.hda[s][slot] = make_float4((float)(box.cx - 2.0 * h.x), (float)(box.cy - 2.0 * h.y),
                                                 (float)(box.cx - 2.0 * h.z), (float)(box.cy - 2.0 * h.w));
                } else if constexpr (VEL == VK_CONST && (WGT & 3) == 2) {
                    // the true-amplitude kernels take the legs relative to the tile centre: FP64 legs
                    // at the tile centre c, R_ac = |c - a|, and tau_c = (R_sc + R_rc) / (v0 dt) - t0/dt
                    {
                    const double esx = __dadd_rn(box.cx, -(double)h.x), esy = __dadd_rn(box.cy, -(double)h.y);
                    const double erx = __dadd_rn(box.cx, -(double)h.z), ery = __dadd_rn(box.cy, -(double)h.w);
                    const double zc2 = __dmul_rn(box.cz, box.cz);
                    const double rsc = __dsqrt_rn(__dadd_rn(__dadd_rn(__dmul_rn(esx, esx), __dmul_rn(esy, esy)), zc2));
                    const double rrc = __dsqrt_rn(__dadd_rn(__dadd_rn(__dmul_rn(erx, erx), __dmul_rn(ery, ery)), zc2));
                    tau_ref = __dadd_rn(tau_ref, __ddiv_rn(__dadd_rn(rsc, rrc), __dmul_rn(g.v0, g.dtd)));
                    S.refs[s][slot] = make_float4((float)rsc, (float)rrc, 0.f, 0.f);
                    S.hda[s][slot] = make_float4((float)(box.cx - 2.0 * h.x), (float)(box.cy - 2.0 * h.y),
                                                 (float)(box.cx - 2.0 * h.z), (float)(box.cy - 2.0 * h.w));
                    }
                } else if constexpr (VEL == VK_PSTM) {
                    // FP64 legs at the tile centre (x_c, t0_c): R_ac = sqrt(|c - a|^2 + ze_c^2) on the
                    // straight rays of the RMS medium, and tau_c = C1(t0_c) (R_sc + R_rc) - t0/dt
                    const double esx = __dadd_rn(box.cx, -(double)h.x), esy = __dadd_rn(box.cy, -(double)h.y);
                    const double erx = __dadd_rn(box.cx, -(double)h.z), ery = __dadd_rn(box.cy, -(double)h.w);
                    const double rsc = __dsqrt_rn(__dadd_rn(__dadd_rn(__dmul_rn(esx, esx), __dmul_rn(esy, esy)), pt.pze2));
                    const double rrc = __dsqrt_rn(__dadd_rn(__dadd_rn(__dmul_rn(erx, erx), __dmul_rn(ery, ery)), pt.pze2));
                    const double sc = __dadd_rn(rsc, rrc);
                    tau_ref = __dadd_rn(tau_ref, __dmul_rn(pt.pc1, sc));
                    S.refs[s][slot] = make_float4((float)rsc, (float)rrc, (float)sc, 0.f);
                    S.hda[s][slot] = make_float4((float)(box.cx - 2.0 * h.x), (float)(box.cy - 2.0 * h.y),
                                                 (float)(box.cx - 2.0 * h.z), (float)(box.cy - 2.0 * h.w));
                }
                S.hdr[s][slot] = h;
                S.mid[s][slot] = m;
                S.tb[s][slot] = (float)__dadd_rn(__dmul_rn((double)lo, g.dtd), g.t0d);
                // every column of the tile inside the aperture: the column test is monotone in
                // |column - midpoint| per axis, so the corner farthest on both axes decides it
                bool whole = false;
                if (g.use_aperture) {
                    const float ex = fmaxf(fabsf(__fsub_rn(box.xlo, m.x)), fabsf(__fsub_rn(box.xhi, m.x)));
                    const float ey = fmaxf(fabsf(__fsub_rn(box.ylo, m.y)), fabsf(__fsub_rn(box.yhi, m.y)));
                    whole = __fadd_rn(__fmul_rn(ex, ex), __fmul_rn(ey, ey)) <= (g.use_taper ? g.ap_core2 : g.A2);
                }
                const float lim = (float)(hi - lo);
                // w: c_half, its sign bit set when the window was not clipped at 0 or nt - 1 (then
                // every point of the tile box has 0 <= tau - lo <= hi - lo by construction)
                S.win[s][slot] = make_int4(__float_as_int((float)(tau_ref - (double)lo)),
                                           dst + (lo - lo_al) - MAGIC_BITS,
                                           __float_as_int(0.5f * lim) | (whole ? (int)0x80000000 : 0),
                                           __float_as_int(0.5f * lim + EDGE_EPS) | (clipped ? 0 : (int)0x80000000));
            }
            if (lane == 0 && bytes > 0) mbar_expect_tx(&S.full[s], (uint32_t)bytes);
            __syncwarp();
            if (fits) {
                const int j = tr.perm[k];
                const TT* src = traces + (long long)j * g.ld + lo_al;
                bulk_g2s(data + s * cap + used + excl, src, (uint32_t)(len_al * g.esize), &S.full[s]);
            }
            cnt += nfit;
            used += used_add;
            cur += consumed;
            if (lane == 0) {
                S.stat[0] += (unsigned)consumed;
                S.stat[1] += (unsigned)nfit;
            }
            if (cur >= te && tr.cell_start) next_row(S.row, S.rng, cur, te);   // the tile's next cell row
            full = (nofit != 0u) || cnt >= BMAX;
        }
        __syncwarp();
        if (lane == 0) {
            S.cnt[s] = cnt;
            S.last[s] = (cur >= te) ? 1 : 0;
            mbar_arrive(&S.full[s]);
        }
        __syncwarp();
        ++n;
        if (cur >= te) break;
    }
    if (wc.stats && lane == 0) {
        atomicAdd(&wc.stats[0], (unsigned long long)S.stat[0]);
        atomicAdd(&wc.stats[1], (unsigned long long)S.stat[1]);
        atomicAdd(&wc.stats[2], 1ull);
    }
    if (failed) {
        if (lane == 0) atomicOr(wc.status, 1);
        // let every copy already issued land before the CTA can exit
        const int first = n - STAGES > n_begin ? n - STAGES : n_begin;
        for (int f = first; f < n; ++f)
            mbar_wait_bounded(&S.full[f % STAGES], (f / STAGES) & 1, 0, WAIT_NS, nullptr);
    }
    return n;
}

// Column (tx, ty) and z-group of consumer thread `tid` in the tile.  When the layer's footprint
// allows it, a warp covers an 8 x 4 block of columns instead of 32 x 1 or 16 x 2: a compact
// footprint leaves fewer lanes idle where the aperture boundary crosses the warp.  Each half warp, the
// lanes that an 8-byte shared load serves together, covers 4 x 4 of them: the samples they read lie
// within fewer banks' turns (3D time migration 11.67 -> 11.34 ms).
__device__ __forceinline__ void thread_column(const TileShape& ts, int tid, int& tx, int& ty, int& tzg)
{
    const int layer = ts.cx * ts.cy;
    tzg = tid / layer;
    const int r = tid - tzg * layer;
    if ((ts.cx & 7) == 0 && (ts.cy & 3) == 0) {
        const int wl = r >> 5, lane = r & 31, bx = ts.cx >> 3;
        tx = (wl % bx) * 8 + (lane & 3) + 4 * (lane >> 4);
        ty = (wl / bx) * 4 + ((lane >> 2) & 3);
    } else {
        tx = r % ts.cx;
        ty = r / ts.cx;
    }
}

// ------------------------------------------------------------------ consumer warps
// `n`: stages consumed before this tile (see mig_producer); returns the new count.
//
// Depths are taken in pairs: every FP32 operation but the roots, reciprocals and sample reads is a
// packed one (kh_f32x2.cuh), so that a contribution takes about half the issue slots on the FMA
// pipe.  The per-depth constants are laid out for it ((x0, x1, y0, y1), (z0, z1, w0, w1) per pair).
// Against one depth at a time: 36.1 -> 22.2 instructions per contribution on the 2.5D line (20 000
// traces, 512 x 400: 5.67 -> 4.68 ms), 1.69 -> 1.47 s for 100 000 traces into 256^3, the same
// bits.  That left shared-memory wavefronts (61-97 % of their peak: the source leg's 16 bytes a lane and
// pair took a third) and the one dependent chain a warp has in flight.  So two traces of one source
// position are taken together where both are unchecked: the source leg and the per-depth constants are
// read once for both, the two chains overlap, and each point still adds them in order: 3D time
// migration 14.5 -> 11.3 ms, 1.47 -> 1.39 s for 256^3, the 2.5D line 4.30 -> 4.06 ms, the same bits.  What
// bounds it now: the 60-65 % of issue slots and of the MUFU's cycles that four warps a scheduler reach
// at 96 registers.  Tried and dropped: one reciprocal for a pair's two (0-4 % slower), byte offsets into
// the ring (0-3 %), partial unrolls (3-15 %), one trace of the next pair ahead (0-1 %).
//
// Linear v(z): the source leg of a contribution depends only on the column and the source
// position, and traces of one bin arrive shot by shot (the bin sort is stable), so each thread
// keeps (C1 ln(1 + rho_s), sqrt(q_s)) of its 16 depths for the current source in `srcc` (its
// own slots, [pair * CONSUMERS + tid]) and recomputes them only when the (warp-uniform) source
// changes.  tau - lo = c0rel + C1 ln(1 + rho_s) + C1 ln(1 + rho_r) with c0rel = tau_ref - lo,
// each leg's logarithm from the per-leg fit (LPT = its length).  The weight's gamma(z)
// multiplies each depth's sum once, before the store.
// Adds a column's depths to the parts before: the sum that k_split_sum forms, in the same order.  A call for
// linear v(z), where these lines in the kernel cost every launch 0.5 % (10 000 traces into 256^3: 140.5 -> 141.1
// ms), and in the kernel else, where the call costs (radial tables 1.5 %).
__device__ __forceinline__ void add_column_here(float* out, int n, float4 a, float4 b, float4 c, float4 d)
{
    const float v[16] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w, c.x, c.y, c.z, c.w, d.x, d.y, d.z, d.w};
#pragma unroll
    for (int i = 0; i < 16; ++i)
        if (i < n) out[i] = __fadd_rn(out[i], v[i]);
}
__device__ __noinline__ static void add_column(float* out, int n, float4 a, float4 b, float4 c, float4 d)
{
    add_column_here(out, n, a, b, c, d);
}

template <int VEL, int WGT, bool FAST, typename TT, int LPT, typename TB>
__device__ __forceinline__ int mig_consumer(MigSmem& S, const TT* data, const GeomParams& g,
                                            const TileShape& ts, int x0, int y0, int z0,
                                            const TileBox& box, int bin, float* __restrict__ image,
                                            const WaitCfg& wc, const TB* tab, float2* srcc, int cap, int n)
{
    constexpr int WB = WGT & 3;                 // the weight (KH_W_*)
    constexpr bool AA = (WGT & W_AA) != 0;      // operator anti-aliasing compiled in
    constexpr int NP = NZ / 2;                  // depth pairs
    using T_ = std::true_type;
    using F_ = std::false_type;
    const int tid = threadIdx.x, lane = tid & 31;
    int tx, ty, tzg;
    thread_column(ts, tid, tx, ty, tzg);
    const int ix = x0 + tx, iy = y0 + ty, izb = z0 + tzg * NZ;
    const bool col_ok = ix < g.nx && iy < g.ny && izb < g.nz;
    const float cxf = col_coord(g.ox, ix, g.dx);
    const float cyf = (g.dim == 3) ? col_coord(g.oy, iy, g.dy) : 0.f;
    const double xd = grid_coord(g.ox, ix, g.dx), yd = (g.dim == 3) ? grid_coord(g.oy, iy, g.dy) : 0.0;
    const float dxc = (float)(xd - box.cx), dyc = (float)(yd - box.cy);
    const ulonglong2* zc = reinterpret_cast<const ulonglong2*>(&S.zc[tzg * NZ]);   // per pair: zc[2p], zc[2p + 1]
    const float* zg = &S.z2[tzg * NZ];   // depth factor of the weight
    const int zero_off = (int)(((const char*)S.zero - (const char*)data) / (int)sizeof(TT));

    F2 acc[NP];
#pragma unroll
    for (int p = 0; p < NP; ++p) acc[p] = f2(0.f);
    // the source cache: two values a depth, or one where the weight needs none of the source leg (then
    // 8-byte slots: 16-byte ones would be read with a two-way bank conflict)
    constexpr bool SV1 = (VEL == VK_LINEAR || VEL == VK_PSTM) && WB == 0;
    ulonglong2* my_src2 = reinterpret_cast<ulonglong2*>(srcc) + tid;
    F2* my_src1 = reinterpret_cast<F2*>(srcc) + tid;
    auto set_src = [&](int p, F2 a, F2 b) {
        if constexpr (SV1) my_src1[p * CONSUMERS] = a;
        else my_src2[p * CONSUMERS] = make_ulonglong2(a, b);
    };
    auto get_src = [&](int p) -> ulonglong2 {
        if constexpr (SV1) return make_ulonglong2(my_src1[p * CONSUMERS], 0ull);
        else return my_src2[p * CONSUMERS];
    };
    unsigned psx = 0xffffffffu, psy = 0xffffffffu;   // source of the cached leg (NaN bits: none)
    const TT* ring = data - LEAD;
    const unsigned ring_last = (unsigned)(LEAD + STAGES * cap + SLACK - 2);   // the kernel's ring
    const bool zfull = izb + NZ <= g.nz;   // all 16 depths of this thread lie in the grid
    // anti-aliasing: the range [aa_lo, aa_hi] of z^2 over the thread's depths (constant velocity)
    // or of z (v0 + k z, with the thread's first depth aa_z0 and the depth step aa_dz)
    float aa_lo = 0.f, aa_hi = 0.f, aa_z0 = 0.f, aa_dz = 0.f;
    if constexpr (AA) {
        aa_z0 = (float)grid_coord(g.oz, izb, g.dz);
        aa_dz = (float)g.dz;
        const float zl = (float)grid_coord(g.oz, izb + NZ - 1, g.dz);
        if constexpr (VEL == VK_CONST) {
            aa_lo = (aa_z0 <= 0.f && zl >= 0.f) ? 0.f : fminf(aa_z0 * aa_z0, zl * zl);
            aa_hi = fmaxf(aa_z0 * aa_z0, zl * zl);
        } else {
            aa_lo = fminf(aa_z0, zl);
            aa_hi = fmaxf(aa_z0, zl);
        }
    }
    // gridded model: the column's node column and fraction, and its first node row (threads
    // whose depths all lie below the image read the last rows)
    const float* gcol = nullptr;
    float gfx = 0.f;
    if constexpr (VEL == VK_GRID) {
        const int gi = grid_col(g, ix, &gfx);
        const int jb = min(g.gzoff + izb / LPT, g.gnz - (NZ / LPT + 1));
        gcol = g.gtab + (long long)jb * g.gnx + gi;
    }
    // gridded model: the receiver table nodes of the next trace of the stage, read one trace
    // ahead so that their L2 latency overlaps this trace's depth loop (pf_t: the trace they
    // belong to, -1: none); not with nodes at every depth (17 nodes per column would spill)
    constexpr bool GPF = (VEL == VK_GRID) && (NZ / LPT + 1) <= 9;
    constexpr int GK = GPF ? NZ / LPT + 1 : 1;
    float pfa[GK], pfb[GK];
    int pf_t = -1;

    bool failed = false;
    while (true) {
        const int s = n % STAGES;
        if (!warp_wait(&S.full[s], (n / STAGES) & 1, wc.polls, wc.ns, wc.status)) {
            failed = true;
            break;
        }
        const int cnt = S.cnt[s];
        const int last = S.last[s];
        pf_t = -1;   // what was read ahead for a skipped trace of the last stage is no trace's of this one
        // a staged trace as this thread sees it
        struct View {
            int4 w;
            float4 h;
            float tp;          // aperture taper of this column (1 in the taper's core)
            bool inside, any;  // the column in the trace's aperture; any of the warp's
            // unclipped window, and every lane inside the aperture (its untapered core, with a
            // taper) with all 16 depths in the grid: every tau is inside the window, no validity
            // test and no taper are needed
            bool unchecked;
        };
        auto view = [&](int t) -> View {
            View v;
            v.w = S.win[s][t];
            v.inside = col_ok;
            v.tp = 1.f;
            if (g.use_aperture && v.w.z >= 0) {   // sign bit of w.z: every column is inside (its core)
                const float2 m = S.mid[s][t];
                v.inside = v.inside && in_aperture(cxf, cyf, m.x, m.y, g.A2);
                if (g.use_taper && v.inside) v.tp = aperture_taper(cxf, cyf, m.x, m.y, g);
            }
            v.any = __any_sync(0xffffffffu, v.inside);
            v.h = S.hdr[s][t];
            v.unchecked = v.w.w < 0 && (!g.use_taper || v.w.z < 0) && __all_sync(0xffffffffu, v.inside && zfull);
            return v;
        };
        for (int t = 0; t < cnt; ++t) {
            const View v = view(t);
            if (!v.any) continue;
            const int4 w = v.w;
            const float4 h = v.h;
            const bool inside = v.inside, unchecked = v.unchecked;
            const float c0rel = __int_as_float(w.x);
            const float cmid = __int_as_float(w.z & 0x7fffffff);
            const float chalf = inside ? __int_as_float(w.w & 0x7fffffff) : -1.f;
            // Two traces at a time where both are unchecked and share the source position (which the
            // constant-velocity legs do not ask for): the per-depth constants and the source leg are read
            // once for both, and their two dependent chains overlap.
            auto second = [&](bool same_source) -> View {
                View u{};
                if (unchecked && t + 1 < cnt) {
                    u = view(t + 1);
                    u.unchecked = u.unchecked && (!same_source || (__float_as_uint(u.h.x) == __float_as_uint(h.x) &&
                                                                   __float_as_uint(u.h.y) == __float_as_uint(h.y)));
                }
                return u;
            };
            // adds a depth pair's samples at th, weighted (W: unless W = 1, where the weight's part
            // here is 1)
            auto add = [&](int p, F2 W, F2 val) {
                if constexpr (WB == 0) acc[p] = add2(acc[p], val);
                else acc[p] = fma2(W, val, acc[p]);
            };
            // the depth loop over one trace, compiled for its class; eval(p, W) gives tau - lo and the weight
            auto single = [&](auto&& eval, auto&& alias_weight, int aacls) {
                auto zloop = [&](auto checked, auto tapered, auto alias) {
#pragma unroll
                    for (int p = 0; p < NP; ++p) {
                        F2 W = 0;
                        const F2 th = eval(p, W);
                        F2 val;
                        if constexpr (decltype(checked)::value)
                            val = sample2_at<TT>(data, th, w.y, cmid, chalf, zero_off);
                        else
                            val = sample2_unchecked<TT>(ring, th, w.y + LEAD, ring_last);
                        if constexpr (decltype(tapered)::value) val = mul2(val, f2(v.tp));
                        if constexpr (decltype(alias)::value) val = mul2(val, alias_weight(p));
                        add(p, W, val);
                    }
                };
                if constexpr (AA) {
                    if (aacls == 2) {
                        if (unchecked) zloop(F_(), F_(), T_());
                        else zloop(T_(), T_(), T_());
                        return;
                    }
                }
                if (unchecked) zloop(F_(), F_(), F_());
                else if (g.use_taper) zloop(T_(), T_(), F_());
                else zloop(T_(), F_(), F_());
            };
            // and over two unchecked ones, in order
            auto both = [&](auto&& eval_a, auto&& eval_b, int base_b) {
#pragma unroll
                for (int p = 0; p < NP; ++p) {
                    F2 Wa = 0, Wb = 0;
                    const F2 ta = eval_a(p, Wa), tb = eval_b(p, Wb);
                    const F2 va = sample2_unchecked<TT>(ring, ta, w.y + LEAD, ring_last);
                    const F2 vb = sample2_unchecked<TT>(ring, tb, base_b + LEAD, ring_last);
                    add(p, Wa, va);
                    add(p, Wb, vb);
                }
            };
            auto no_alias = [](int) -> F2 { return 0; };
            if constexpr (VEL == VK_TABLE || VEL == VK_GRID) {
                // T_s + T_r from tables, in table units: the shared radial table, or the two legs'
                // first-arrival tables (global memory, L2-resident); per leg the profile at the K
                // nodes spanning the thread's 16 depths (one every M samples), then linear in depth.
                // The source leg T_s is cached per source position (its location) like the linear
                // path's
                constexpr int M = LPT;            // depth nodes every M samples (1, 2 or 4)
                constexpr int K = NZ / M + 1;
                F2* my_ts = reinterpret_cast<F2*>(srcc) + tid;
                const float dxs = cxf - h.x, dxr = cxf - h.z;
                const float dys = VEL == VK_GRID ? 0.f : cyf - h.y, dyr = VEL == VK_GRID ? 0.f : cyf - h.w;
                const float dhs2 = fmaf(dxs, dxs, dys * dys), dhr2 = fmaf(dxr, dxr, dyr * dyr);
                // a gridded model's headers carry the locations' indexes in their y slots
                const unsigned kx = VEL == VK_GRID ? 0u : __float_as_uint(h.x), ky = __float_as_uint(h.y);
                if (kx != psx || ky != psy) {   // new source
                    float ps[K];
                    if constexpr (VEL == VK_GRID)
                        grid_profile<K>(gcol + (long long)__float_as_int(h.y) * g.gstride, g.gnx, gfx, ps);
                    else
                        tab_profile<TB, K, FAST>(tab, g, dhs2, izb / M, ps);
#pragma unroll
                    for (int p = 0; p < NP; ++p)
                        my_ts[p * CONSUMERS] = f2(tab_depth<M>(ps, 2 * p), tab_depth<M>(ps, 2 * p + 1));
                    psx = kx;
                    psy = ky;
                }
                float pr[K];
                if constexpr (VEL == VK_GRID) {
                    if (GPF && pf_t == t) {
#pragma unroll
                        for (int k = 0; k < K; ++k) pr[k] = fmaf(gfx, pfb[GPF ? k : 0] - pfa[GPF ? k : 0], pfa[GPF ? k : 0]);
                    } else {
                        grid_profile<K>(gcol + (long long)__float_as_int(h.w) * g.gstride, g.gnx, gfx, pr);
                    }
                    pf_t = -1;
                    if (GPF && t + 1 < cnt) {   // the next trace's receiver nodes, in flight during this loop
                        const int ln = __float_as_int(S.hdr[s][t + 1].w);
                        if (ln >= 0) {
                            const float* c0 = gcol + (long long)ln * g.gstride;
#pragma unroll
                            for (int k = 0; k < GK; ++k) {
                                pfa[k] = __ldg(c0 + k * g.gnx);
                                pfb[k] = __ldg(c0 + k * g.gnx + 1);
                            }
                            pf_t = t + 1;
                        }
                    }
                } else {
                    tab_profile<TB, K, FAST>(tab, g, dhr2, izb / M, pr);
                }
                const F2 c0 = f2(c0rel);
                single([&](int p, F2& W) -> F2 {
                    // w_z multiplies the sum once, at the store
                    if constexpr (WB == 1) {
                        const F2 z2 = zc[2 * p].x;   // z^2
                        W = add2(sqrt2<FAST>(add2(f2(dhs2), z2)), sqrt2<FAST>(add2(f2(dhr2), z2)));
                    }
                    return fma2(add2(my_ts[p * CONSUMERS], f2(tab_depth<M>(pr, 2 * p), tab_depth<M>(pr, 2 * p + 1))), f2(g.C1), c0);
                }, no_alias, 1);
            } else if constexpr (VEL == VK_PSTM) {
                // time migration relative to the tile centre: per leg R_a - R_ac = (q_a - q_ac) /
                // (R_a + R_ac) with q_a - q_ac = dP_a + (ze^2 - ze_c^2), so that
                // tau - lo = c0rel + (C1(t0) - C1(t0_c)) S_c + C1(t0) (dR_s + dR_r) carries only
                // quantities of a few tens of samples; the source leg (dR_s, R_s) is cached per
                // source position like the linear path's
                if (__float_as_uint(h.x) != psx || __float_as_uint(h.y) != psy) {   // new source
                    const float4 a = S.hda[s][t];
                    const F2 rsc = f2(S.refs[s][t].x);
                    const F2 dPs = f2(fmaf(dxc, cxf + a.x, dyc * (cyf + a.y)));
                    const float exs = cxf - h.x, eys = cyf - h.y;
                    const F2 dhs2 = f2(fmaf(exs, exs, eys * eys));
#pragma unroll
                    for (int p = 0; p < NP; ++p) {
                        const ulonglong2 c = zc[2 * p];   // (ze^2, ze^2 - ze_c^2)
                        const F2 R = sqrt2<FAST>(add2(dhs2, c.x));
                        set_src(p, mul2(add2(dPs, c.y), rcp2<FAST>(add2(R, rsc))), R);
                    }
                    psx = __float_as_uint(h.x);
                    psy = __float_as_uint(h.y);
                }
                struct Leg {
                    F2 dP, dh2, rc, sc, c0;
                };
                auto leg = [&](int tt, const View& q) -> Leg {
                    const float4 a = S.hda[s][tt], rf = S.refs[s][tt];   // rf: (R_sc, R_rc, S_c, -)
                    const float ex = cxf - q.h.z, ey = cyf - q.h.w;
                    return Leg{f2(fmaf(dxc, cxf + a.z, dyc * (cyf + a.w))), f2(fmaf(ex, ex, ey * ey)), f2(rf.y), f2(rf.z),
                               f2(__int_as_float(q.w.x))};
                };
                auto eval = [&](const Leg& q) {
                    return [&](int p, F2& W) -> F2 {
                        const ulonglong2 c = zc[2 * p], d = zc[2 * p + 1];   // d: (C1(t0), C1(t0) - C1(t0_c))
                        const ulonglong2 sv = get_src(p);                    // (dR_s, R_s)
                        const F2 R = sqrt2<FAST>(add2(q.dh2, c.x));
                        const F2 dR = mul2(add2(q.dP, c.y), rcp2<FAST>(add2(R, q.rc)));
                        // W = w_z (R_s + R_r); w_z multiplies the sum once, at the store
                        if constexpr (WB == 1) W = add2(sv.y, R);
                        return fma2(d.x, add2(sv.x, dR), fma2(d.y, q.sc, q.c0));
                    };
                };
                const Leg qa = leg(t, v);
                const View u = second(true);
                if (u.unchecked) {
                    const Leg qb = leg(t + 1, u);
                    both(eval(qa), eval(qb), u.w.y);
                    ++t;
                } else {
                    single(eval(qa), no_alias, 1);
                }
            } else if constexpr (VEL == VK_CONST && WB != 2) {
                struct Leg {
                    F2 dhs2, dhr2, c0;
                };
                auto leg = [&](const View& q) -> Leg {
                    const float dxs = cxf - q.h.x, dys = cyf - q.h.y, dxr = cxf - q.h.z, dyr = cyf - q.h.w;
                    return Leg{f2(fmaf(dxs, dxs, dys * dys)), f2(fmaf(dxr, dxr, dyr * dyr)), f2(__int_as_float(q.w.x))};
                };
                auto eval = [&](const Leg& q) {
                    return [&](int p, F2& W) -> F2 {
                        const F2 z2 = zc[2 * p].x;   // z^2
                        const F2 Ssum = add2(sqrt2<FAST>(add2(q.dhs2, z2)), sqrt2<FAST>(add2(q.dhr2, z2)));
                        W = Ssum;   // w_z multiplies the sum once, at the store
                        return fma2(Ssum, f2(g.C1), fma2(Ssum, f2(g.C1lo), q.c0));
                    };
                };
                const Leg qa = leg(v);
                if constexpr (AA) {
                    // anti-aliasing: skip a trace whose every weight here is 0; evaluate the weight
                    // per contribution only where the warp's depth range holds weights below 1
                    const float dxs = cxf - h.x, dys = cyf - h.y, dxr = cxf - h.z, dyr = cyf - h.w;
                    const int aacls = aa_class(g.aa_c, dxs, dys, dxr, dyr, aa_lo, aa_hi, inside);
                    if (aacls == 0) continue;
                    single(eval(qa), [&](int p) -> F2 {
                        const F2 z2 = zc[2 * p].x;
                        const float2 s2 = f2_get(sqrt2<FAST>(add2(qa.dhs2, z2))), r2 = f2_get(sqrt2<FAST>(add2(qa.dhr2, z2)));
                        return f2(aa_weight<FAST>(g.aa_c, dxs, dys, dxr, dyr, s2.x, r2.x),
                                  aa_weight<FAST>(g.aa_c, dxs, dys, dxr, dyr, s2.y, r2.y));
                    }, aacls);
                } else {
                    const View u = second(false);
                    if (u.unchecked) {
                        const Leg qb = leg(u);
                        both(eval(qa), eval(qb), u.w.y);
                        ++t;
                    } else {
                        single(eval(qa), no_alias, 1);
                    }
                }
            } else if constexpr (VEL == VK_CONST) {
                // the true-amplitude weight: each leg relative to the tile centre: R_a - R_ac =
                // (q_a - q_ac) / (R_a + R_ac) with q_a - q_ac = dP_a + (z^2 - z_c^2), so tau - lo =
                // c0rel + C1 (dR_s + dR_r) carries only quantities of a few tens of samples (the full
                // two-way time, hundreds of samples, is in the FP64 reference).  One reciprocal root
                // gives 1/R_a and R_a = q_a / R_a; the source leg's (dR_s, 1/R_s) is cached per source
                // position.  The weight z (R_s + R_r) (1/R_s^2 + 1/R_r^2) / 2 (2D: sqrt(R_s R_r)) is 0 on
                // the surface row, where zc's z / 2 is stored as 0 (every factor is finite, see root_pair)
                int aacls = 1;   // anti-aliasing classes as in the direct branch
                if constexpr (AA) {
                    aacls = aa_class(g.aa_c, cxf - h.x, cyf - h.y, cxf - h.z, cyf - h.w, aa_lo, aa_hi, inside);
                    if (aacls == 0) continue;
                }
                const float exs = cxf - h.x, eys = cyf - h.y;
                const F2 dhs2 = f2(fmaf(exs, exs, eys * eys));
                if (__float_as_uint(h.x) != psx || __float_as_uint(h.y) != psy) {   // new source
                    const float4 a = S.hda[s][t];
                    const F2 dPs = f2(fmaf(dxc, cxf + a.x, dyc * (cyf + a.y))), rsc = f2(S.refs[s][t].x);
#pragma unroll
                    for (int p = 0; p < NP; ++p) {
                        const ulonglong2 c = zc[2 * p];   // (z^2, z^2 - z_c^2)
                        F2 R, ir;
                        root_pair<FAST>(add2(dhs2, c.x), R, ir);
                        set_src(p, mul2(add2(dPs, c.y), rcp2<FAST>(max2(add2(R, rsc), 1e-30f))), ir);
                    }
                    psx = __float_as_uint(h.x);
                    psy = __float_as_uint(h.y);
                }
                struct Leg {
                    F2 dP, dh2, rc, c0;
                };
                auto leg = [&](int tt, const View& q) -> Leg {
                    const float4 a = S.hda[s][tt];
                    const float ex = cxf - q.h.z, ey = cyf - q.h.w;
                    return Leg{f2(fmaf(dxc, cxf + a.z, dyc * (cyf + a.w))), f2(fmaf(ex, ex, ey * ey)), f2(S.refs[s][tt].y),
                               f2(__int_as_float(q.w.x))};   // refs: (R_sc, R_rc, -, -)
                };
                F2 ir_last = 0;   // 1/R_r of the depth pair evaluated last
                auto eval = [&](const Leg& q) {
                    return [&](int p, F2& W) -> F2 {
                        const ulonglong2 c = zc[2 * p];
                        const ulonglong2 sv = get_src(p);   // (dR_s, 1/R_s)
                        F2 Rr, ir;
                        root_pair<FAST>(add2(q.dh2, c.x), Rr, ir);
                        if constexpr (AA) ir_last = ir;
                        const F2 dR = mul2(add2(q.dP, c.y), rcp2<FAST>(max2(add2(Rr, q.rc), 1e-30f)));
                        const F2 is = sv.y, qs = add2(dhs2, c.x), Rs = FAST ? mul2(qs, is) : sqrt2<false>(qs);
                        const F2 amp = g.dim == 3 ? add2(Rs, Rr) : sqrt2<FAST>(mul2(Rs, Rr));
                        W = mul2(mul2(zc[2 * p + 1].x, amp), fma2(is, is, mul2(ir, ir)));
                        return fma2(f2(g.C1), add2(sv.x, dR), q.c0);
                    };
                };
                const Leg qa = leg(t, v);
                if constexpr (AA) {
                    const float exr = cxf - h.z, eyr = cyf - h.w;
                    single(eval(qa), [&](int p) -> F2 {
                        const float2 s2 = f2_get(get_src(p).y), r2 = f2_get(ir_last);
                        return f2(aa_weight_r(g.aa_c, exs, eys, exr, eyr, s2.x, r2.x),
                                  aa_weight_r(g.aa_c, exs, eys, exr, eyr, s2.y, r2.y));
                    }, aacls);
                } else {
                    const View u = second(true);
                    if (u.unchecked) {
                        const Leg qb = leg(t + 1, u);
                        both(eval(qa), eval(qb), u.w.y);
                        ++t;
                    } else {
                        single(eval(qa), no_alias, 1);
                    }
                }
            } else {
                int aacls = 1;   // anti-aliasing classes as in the constant-velocity branches
                if constexpr (AA && VEL == VK_LINEAR) {
                    aacls = aa_class_lin(g, cxf - h.x, cyf - h.y, cxf - h.z, cyf - h.w, aa_lo, aa_hi, inside);
                    if (aacls == 0) continue;
                }
                if (__float_as_uint(h.x) != psx || __float_as_uint(h.y) != psy) {   // new source
                    const float4 a = S.hda[s][t];
                    const LegRef2 rs(S.refs[s][t]);
                    const F2 dPs = f2(fmaf(dxc, cxf + a.x, dyc * (cyf + a.y)));
                    const float exs = cxf - h.x, eys = cyf - h.y;
                    const F2 dhs2 = f2(fmaf(exs, exs, eys * eys));
#pragma unroll
                    for (int p = 0; p < NP; ++p) {
                        F2 sqs = 0;
                        const F2 rho_s = leg_delta2<WB, FAST>(dPs, dhs2, zc[2 * p], zc[2 * p + 1], rs, sqs);
                        set_src(p, leg_log2<LPT>(rho_s, g, f2(0.f)), sqs);
                    }
                    psx = __float_as_uint(h.x);
                    psy = __float_as_uint(h.y);
                }
                struct Leg {
                    LegRef2 rr;
                    F2 dP, dh2, c0;
                };
                auto leg = [&](int tt, const View& q) -> Leg {
                    const float4 a = S.hda[s][tt];
                    const float ex = cxf - q.h.z, ey = cyf - q.h.w;
                    return Leg{LegRef2(S.refr[s][tt]), f2(fmaf(dxc, cxf + a.z, dyc * (cyf + a.w))), f2(fmaf(ex, ex, ey * ey)),
                               f2(__int_as_float(q.w.x))};
                };
                auto eval = [&](const Leg& q) {
                    return [&](int p, F2& W) -> F2 {
                        F2 sqr = 0;
                        const ulonglong2 sv = get_src(p);   // (C1 ln(1 + rho_s), sqrt(q_s))
                        const F2 rho_r = leg_delta2<WB, FAST>(q.dP, q.dh2, zc[2 * p], zc[2 * p + 1], q.rr, sqr);
                        // gamma(z) multiplies the sum once, at the store
                        if constexpr (WB == 1) W = add2(sv.y, sqr);
                        return leg_log2<LPT>(rho_r, g, add2(q.c0, sv.x));
                    };
                };
                const Leg qa = leg(t, v);
                if constexpr (AA) {
                    const float exs = cxf - h.x, eys = cyf - h.y, exr = cxf - h.z, eyr = cyf - h.w;
                    const float hs2 = fmaf(exs, exs, eys * eys), hr2 = fmaf(exr, exr, eyr * eyr);
                    single(eval(qa), [&](int p) -> F2 {
                        // each leg's slowness factor at this depth (FP32 geometry: the weight
                        // is flat where rounding could move it)
                        float aw[2];
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            const float zi = fmaf((float)(2 * p + e), aa_dz, aa_z0);
                            const float vv = fmaf(g.aa_v0k, zi, g.aa_v0sq);
                            aw[e] = aa_weight_r(g.aa_c, exs, eys, exr, eyr, aa_leg_lin(fmaf(zi, zi, hs2), vv, g.aa_kq),
                                                aa_leg_lin(fmaf(zi, zi, hr2), vv, g.aa_kq));
                        }
                        return f2(aw[0], aw[1]);
                    }, aacls);
                } else {
                    const View u = second(true);
                    if (u.unchecked) {
                        const Leg qb = leg(t + 1, u);
                        both(eval(qa), eval(qb), u.w.y);
                        ++t;
                    } else {
                        single(eval(qa), no_alias, 1);
                    }
                }
            }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&S.empty[s]);
        ++n;
        if (last) break;
    }
    if (failed) {
        if (lane == 0) atomicOr(wc.status, 1);
        return n;
    }
    if (!col_ok) return n;
    float* out = image + (((long long)bin * g.ny + iy) * g.nx + ix) * (long long)g.nz + izb;
    const bool vec = ((g.nz & 3) == 0) && (izb + NZ <= g.nz) &&
                     ((reinterpret_cast<uintptr_t>(image) & 15) == 0);
    if (ts.seq > 1) {   // a part of its own launch
        float4 q[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float2 a = f2_get(acc[2 * i]), b = f2_get(acc[2 * i + 1]);
            q[i] = make_float4(a.x, a.y, b.x, b.y);
            if constexpr (WB == 1)
                q[i] = make_float4(a.x * zg[4 * i], a.y * zg[4 * i + 1], b.x * zg[4 * i + 2], b.y * zg[4 * i + 3]);
        }
        if constexpr (VEL == VK_LINEAR) add_column(out, g.nz - izb, q[0], q[1], q[2], q[3]);
        else add_column_here(out, g.nz - izb, q[0], q[1], q[2], q[3]);
        return n;
    }
#pragma unroll
    for (int i = 0; i < NZ; i += 4) {
        float2 a = f2_get(acc[i / 2]), b = f2_get(acc[i / 2 + 1]);
        if constexpr (WB == 1) {
            a = make_float2(a.x * zg[i], a.y * zg[i + 1]);
            b = make_float2(b.x * zg[i + 2], b.y * zg[i + 3]);
        }
        if (vec) {
            *reinterpret_cast<float4*>(out + i) = make_float4(a.x, a.y, b.x, b.y);
        } else {
            if (izb + i < g.nz) out[i] = a.x;
            if (izb + i + 1 < g.nz) out[i + 1] = a.y;
            if (izb + i + 2 < g.nz) out[i + 2] = b.x;
            if (izb + i + 3 < g.nz) out[i + 3] = b.y;
        }
    }
    return n;
}

// ------------------------------------------------------------------ gradient consumer
// dB/d(v0, k) of B(m, D) = <m, migrate(D)>: per contribution W m (D[i+1] - D[i]) dT/dth,
// with dT/dth summed over both legs (the 1/dt of dtau/dth is applied in the final sum):
//   constant v:  dT/dv0 = -(R_s + R_r)/v0^2;
//   linear v(z): with q/w = sqrt(q/(q+2)) per leg and vz = v0 + k z,
//                dT/dv0 = -(q/w)_sum (1/v0 + 1/vz)/|k|,
//                dT/dk  = -sgn(k) (T_s + T_r)/|k| + (q/w)_sum (2/k - z/vz)/|k|.
// The traces arrive as slope rows D[i+1] - D[i] (one read per contribution).  Linear v(z): the
// source leg (its logarithm term, q/w and sqrt(q)) is cached per source position as in the
// migration, and tau - lo adds the per-leg logarithms.  Two depths an instruction (packed FP32);
// whole windows skip the validity test where the warp's columns and depths lie in the grid.  Each
// thread sums its 16 z in FP32 per (column, trace) and carries FP64 totals, scaled by the common
// factors (-1/v0^2, 1/|k|) at the end; per-warp FP64 partials go to `partial` for a fixed-order
// final sum.  Issue bounded it with one depth an instruction (80 % active, 56.5 instructions a
// contribution): 10 000 traces into 256^3 264 -> 197 ms, 569 -> 764 G contributions/s, the loop over
// depth pairs unrolled whole (721 unrolled by 4 or 2); 28.8 instructions now, 55 % active, waiting on
// each depth pair's own chain.
template <int VEL, int WGT, bool FAST, typename TT, int LPT>
__device__ void vg_consumer(MigSmem& S, const TT* data, const GeomParams& g, const TileShape& ts,
                            int x0, int y0, int z0, const TileBox& box, int bin,
                            const float* __restrict__ image, double* __restrict__ partial,
                            const WaitCfg& wc, float2* srcc, int cap)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int tx, ty, tzg;
    thread_column(ts, tid, tx, ty, tzg);
    const int ix = x0 + tx, iy = y0 + ty, izb = z0 + tzg * NZ;
    const bool col_ok = ix < g.nx && iy < g.ny;
    const float cxf = col_coord(g.ox, ix, g.dx);
    const float cyf = (g.dim == 3) ? col_coord(g.oy, iy, g.dy) : 0.f;
    const double xd = grid_coord(g.ox, ix, g.dx), yd = (g.dim == 3) ? grid_coord(g.oy, iy, g.dy) : 0.0;
    const float dxc = (float)(xd - box.cx), dyc = (float)(yd - box.cy);
    constexpr int NP = NZ / 2;   // depth pairs
    const ulonglong2* zc = reinterpret_cast<const ulonglong2*>(&S.zc[tzg * NZ]);
    const float* zg = &S.z2[tzg * NZ];   // obliquity: depth factor (linear: gamma(z)), folded into the image value
    const int zero_off = (int)(((const char*)S.zero - (const char*)data) / (int)sizeof(TT));
    const TT* ring = data - LEAD;
    const unsigned ring_last = (unsigned)(LEAD + STAGES * cap + SLACK - 1);
    const bool in_grid = __all_sync(0xffffffffu, col_ok && izb + NZ <= g.nz);
    const float dtf = (float)g.dtd;
    const float inv_v0 = (float)(1.0 / g.v0);
    const float sgnk = g.k < 0.0 ? -1.f : 1.f;
    const float two_over_k = (VEL == VK_LINEAR) ? (float)(2.0 / g.k) : 0.f;
    const float inv_a = (VEL == VK_LINEAR) ? (float)(1.0 / g.a) : 0.f;
    const float zb = (float)(g.oz + izb * g.dz), dzf = (float)g.dz;

    // per thread and depth pair in shared memory: the image values times the weight's depth factor,
    // and for linear v(z) the source-leg cache (C1 ln(1 + rho_s), (q/w)_s) and sqrt(q_s)
    F2* my_mv = reinterpret_cast<F2*>(srcc) + tid;
    ulonglong2* my_lq = reinterpret_cast<ulonglong2*>(srcc + NP * CONSUMERS) + tid;
    F2* my_sq = reinterpret_cast<F2*>(srcc) + 3 * NP * CONSUMERS + tid;
#pragma unroll
    for (int p = 0; p < NP; ++p) {
        float m[2];
        for (int e = 0; e < 2; ++e) {
            const int i = 2 * p + e;
            m[e] = (col_ok && izb + i < g.nz)
                       ? image[(((long long)bin * g.ny + iy) * g.nx + ix) * (long long)g.nz + izb + i]
                       : 0.f;
            if (WGT == 1) m[e] *= zg[i];
        }
        my_mv[p * CONSUMERS] = f2(m[0], m[1]);
    }
    double G0 = 0.0, G1 = 0.0;
    unsigned psx = 0xffffffffu, psy = 0xffffffffu;

    bool failed = false;
    int n = 0;
    while (true) {
        const int s = n % STAGES;
        if (!warp_wait(&S.full[s], (n / STAGES) & 1, wc.polls, wc.ns, wc.status)) {
            failed = true;
            break;
        }
        const int cnt = S.cnt[s];
        const int last = S.last[s];
        for (int t = 0; t < cnt; ++t) {
            const int4 w = S.win[s][t];
            bool inside = col_ok;
            float tp = 1.f;   // aperture taper of this column
            if (g.use_aperture && w.z >= 0) {   // sign bit of w.z: every column is inside (its core)
                const float2 m = S.mid[s][t];
                inside = inside && in_aperture(cxf, cyf, m.x, m.y, g.A2);
                if (g.use_taper && inside) tp = aperture_taper(cxf, cyf, m.x, m.y, g);
            }
            if (!__any_sync(0xffffffffu, inside)) continue;
            const float c0rel = __int_as_float(w.x);
            const float cmid = __int_as_float(w.z & 0x7fffffff);
            const float chalf = inside ? __int_as_float(w.w & 0x7fffffff) : -1.f;
            const float4 h = S.hdr[s][t];
            F2 g0 = 0, g1 = 0;
            // W m (D[i+1] - D[i]) of a depth pair at th = tau - lo
            auto term = [&](int p, F2 th, F2 W, auto checked) -> F2 {
                float2 d;
                if constexpr (decltype(checked)::value) {
                    const float2 tv = f2_get(th);
                    const bool ok0 = fabsf(tv.x - cmid) <= chalf, ok1 = fabsf(tv.y - cmid) <= chalf;
                    const float2 tm = f2_get(add2_rd(max2(th, 0.f), f2(MAGIC)));   // MAGIC + floor(th), th >= 0
                    d.x = to_f32<TT>(data[ok0 ? __float_as_int(tm.x) + w.y : zero_off]);
                    d.y = to_f32<TT>(data[ok1 ? __float_as_int(tm.y) + w.y : zero_off]);
                } else {   // every tau of the tile box lies in the window; the clamp keeps any read in the ring
                    const float2 tm = f2_get(add2_rd(th, f2(MAGIC)));
                    d.x = to_f32<TT>(ring[min((unsigned)(__float_as_int(tm.x) + w.y + LEAD), ring_last)]);
                    d.y = to_f32<TT>(ring[min((unsigned)(__float_as_int(tm.y) + w.y + LEAD), ring_last)]);
                }
                const F2 ms = mul2(my_mv[p * CONSUMERS], f2(d.x, d.y));
                return WGT == 1 ? mul2(W, ms) : ms;
            };
            if constexpr (VEL == VK_CONST) {
                const float dxs = cxf - h.x, dys = cyf - h.y;
                const float dxr = cxf - h.z, dyr = cyf - h.w;
                const F2 dhs2 = f2(fmaf(dxs, dxs, dys * dys));
                const F2 dhr2 = f2(fmaf(dxr, dxr, dyr * dyr));
                auto zloop = [&](auto checked) {
#pragma unroll
                    for (int p = 0; p < NP; ++p) {
                        const F2 zz = zc[2 * p].x;
                        const F2 S2 = add2(sqrt2<FAST>(add2(dhs2, zz)), sqrt2<FAST>(add2(dhr2, zz)));
                        const F2 th = fma2(S2, f2(g.C1), fma2(S2, f2(g.C1lo), f2(c0rel)));
                        g0 = fma2(term(p, th, S2, checked), S2, g0);
                    }
                };
                if (in_grid && w.w < 0) zloop(std::false_type());
                else zloop(std::true_type());
            } else {
                const float4 rr = S.refr[s][t], a = S.hda[s][t];
                if (__float_as_uint(h.x) != psx || __float_as_uint(h.y) != psy) {   // new source
                    const LegRef2 rs(S.refs[s][t]);
                    const F2 dPs = f2(fmaf(dxc, cxf + a.x, dyc * (cyf + a.y)));
                    const float exs = cxf - h.x, eys = cyf - h.y;
                    const F2 dhs2 = f2(fmaf(exs, exs, eys * eys));
#pragma unroll 2
                    for (int p = 0; p < NP; ++p) {
                        F2 sqs, qws;
                        const F2 rho_s = leg_delta_grad2<FAST>(dPs, dhs2, zc[2 * p], zc[2 * p + 1], rs, sqs, qws);
                        my_lq[p * CONSUMERS] = make_ulonglong2(leg_log2<LPT>(rho_s, g, f2(0.f)), qws);
                        my_sq[p * CONSUMERS] = sqs;
                    }
                    psx = __float_as_uint(h.x);
                    psy = __float_as_uint(h.y);
                }
                const F2 dPr = f2(fmaf(dxc, cxf + a.z, dyc * (cyf + a.w)));
                const float exr = cxf - h.z, eyr = cyf - h.w;
                const F2 dhr2 = f2(fmaf(exr, exr, eyr * eyr));
                const LegRef2 r2(rr);
                const F2 c2 = f2(c0rel);
                // sgn(k) (T_s + T_r) = th sdt + stb
                const F2 sdt = f2(-sgnk * dtf), stb = f2(-sgnk * S.tb[s][t]);
                auto zloop = [&](auto checked) {
#pragma unroll
                    for (int p = 0; p < NP; ++p) {
                        const ulonglong2 za = zc[2 * p];   // (alpha, alpha kappa) of two depths
                        F2 sqr, qwr;
                        const F2 rho_r = leg_delta_grad2<FAST>(dPr, dhr2, za, zc[2 * p + 1], r2, sqr, qwr);
                        const ulonglong2 lq = my_lq[p * CONSUMERS];   // (C1 ln(1 + rho_s), (q/w)_s)
                        const F2 th = leg_log2<LPT>(rho_r, g, add2(c2, lq.x));
                        const F2 wms = term(p, th, WGT == 1 ? add2(my_sq[p * CONSUMERS], sqr) : F2(0), checked);
                        const F2 inv_vz = mul2(za.x, f2(inv_a));
                        const F2 mz = f2(-fmaf((float)(2 * p), dzf, zb), -fmaf((float)(2 * p + 1), dzf, zb));
                        const F2 qw = add2(lq.y, qwr);
                        // |k| dT/dk = (q/w)(2/k - z/vz) - sgn(k) (T_s + T_r); -|k| dT/dv0 = (q/w)(1/v0 + 1/vz)
                        const F2 dk = fma2(qw, fma2(mz, inv_vz, f2(two_over_k)), fma2(th, sdt, stb));
                        g0 = fma2(wms, mul2(qw, add2(f2(inv_v0), inv_vz)), g0);
                        g1 = fma2(wms, dk, g1);
                    }
                };
                if (in_grid && w.w < 0) zloop(std::false_type());
                else zloop(std::true_type());
            }
            if (inside) {   // a lane outside the aperture takes nothing of what it read
                const float2 a0 = f2_get(g0), a1 = f2_get(g1);
                G0 += (double)((a0.x + a0.y) * tp);
                G1 += (double)((a1.x + a1.y) * tp);
            }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&S.empty[s]);
        ++n;
        if (last) break;
    }
    const double inv_ka = (VEL == VK_LINEAR) ? 1.0 / g.kabs : 0.0;
    G0 *= VEL == VK_LINEAR ? -inv_ka : -1.0 / (g.v0 * g.v0);
    G1 *= inv_ka;
    if (failed) {
        if (lane == 0) atomicOr(wc.status, 1);
        G0 = 0.0;
        G1 = 0.0;
    }
    for (int o = 16; o > 0; o >>= 1) {
        G0 += __shfl_xor_sync(0xffffffffu, G0, o);
        G1 += __shfl_xor_sync(0xffffffffu, G1, o);
    }
    if (lane == 0) {
        const long long slot =
            (((long long)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x) * CONSUMER_WARPS + warp;
        partial[2 * slot] = G0;
        partial[2 * slot + 1] = G1;
    }
}

// Per-z constants of a tile's depth range [z0, z0 + cz NZ), written by all threads, per depth pair as
// (x0, x1, y0, y1), (z0, z1, w0, w1).
template <int VEL>
__device__ __forceinline__ void tile_z_setup(MigSmem& S, const GeomParams& g, const TileShape& ts, int z0,
                                             const TileBox& box)
{
    for (int i = threadIdx.x; i < ts.cz * NZ; i += blockDim.x) {
        const double z = grid_coord(g.oz, z0 + i, g.dz);
        const bool off = fabs(z) >= 1e-6 * fabs(g.dz);   // off the surface row, where the weights are 0
        float4 c;
        float zw;
        if constexpr (VEL == VK_LINEAR) {
            c = z_constants_m(z, box.cz, g, zw);
        } else if constexpr (VEL == VK_TABLE || VEL == VK_GRID) {
            c = make_float4((float)(z * z), 0.f, 0.f, 0.f);
            zw = (g.weight == 1 && off) ? (float)(z * g.wscale) : 0.f;
        } else if constexpr (VEL == VK_PSTM) {
            // time migration: z is the two-way vertical time t0; the leg is the straight ray of
            // the RMS velocity, R = sqrt(h^2 + ze^2) with ze = v_rms t0 / 2, and
            // tau = (R_s + R_r) C1(t0) - t0/dt with C1(t0) = 1 / (v_rms dt); stored relative to the
            // tile centre: (ze^2, ze^2 - ze_c^2, C1(t0), C1(t0) - C1(t0_c)), and w_z = ze / (2 r0^2)
            const PstmTile pt = pstm_tile(g, box);
            const double vr = sqrt(vrms2_of(g.v0, g.pk, z));
            const double ze = 0.5 * vr * z;
            const double c1 = 1.0 / (vr * g.dtd);
            c = make_float4((float)(ze * ze), (float)(ze * ze - pt.pze2), (float)c1, (float)(c1 - pt.pc1));
            zw = (g.weight == 1 && off) ? (float)(ze * g.wscale) : 0.f;
        } else {
            // constant velocity: (z^2, z^2 - z_c^2, z / 2 or 0 on the surface row: the factor of the
            // true-amplitude weight), and w_z of the obliquity weight
            const double dq = __dadd_rn(__dmul_rn(z, z), -__dmul_rn(box.cz, box.cz));
            c = make_float4((float)(z * z), (float)dq, off ? 0.5f * (float)z : 0.f, 0.f);
            zw = (g.weight == 1 && off) ? (float)(z * g.wscale) : 0.f;
        }
        S.z2[i] = zw;
        float* d = reinterpret_cast<float*>(&S.zc[i & ~1]) + (i & 1);
        d[0] = c.x;
        d[2] = c.y;
        d[4] = c.z;
        d[6] = c.w;
    }
}

// First sample of part `split`'s image among the partial images of a split launch.
__device__ __forceinline__ long long split_offset(const GeomParams& g, int split)
{
    return (long long)split * g.n_bins * g.ny * g.nx * g.nz;
}

// Shared body of the migration kernel (MODE 0: image out) and of the gradient kernel
// (MODE 1: image in, per-warp partials out).
template <int VEL, int WGT, bool FAST, typename TT, int LPT, int MODE, typename TB = float>
__device__ __forceinline__ void kernel_body(const GeomParams& g, const TileShape& ts, const TraceSet& tr,
                                            const TT* __restrict__ traces, float* __restrict__ image,
                                            int cap, const WaitCfg& wc, double* __restrict__ partial)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    MigSmem& S = *reinterpret_cast<MigSmem*>(smem_raw);
    TT* ring = reinterpret_cast<TT*>(smem_raw + mig_static_bytes());
    TT* data = ring + LEAD;
    __shared__ int s_abort;
    const int bin = blockIdx.y;
    int t = blockIdx.x;
    const int tzi = t % ts.tiles_z;
    t /= ts.tiles_z;
    const int txi = t % ts.tiles_x, tyi = t / ts.tiles_x;
    const int x0 = txi * ts.cx, y0 = tyi * ts.cy, z0 = tzi * ts.cz * NZ;

    const TileBox box = tile_box(g, x0, y0, z0, ts.cx, ts.cy, ts.cz * NZ);

    if (threadIdx.x == 0) {
        // a wait in another CTA of this plan already ran out: results are invalid anyway (the
        // other status bits report skipped inputs, not a stalled launch)
        s_abort = *reinterpret_cast<const volatile int*>(wc.status) & 1;
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&S.full[s], 1);
            mbar_init(&S.empty[s], CONSUMER_WARPS);
        }
        S.zero[0] = S.zero[1] = S.zero[2] = S.zero[3] = 0.f;
        tile_cells(S.row, tr, box);
        fence_barrier_init();
    }
    // per-z constants of the tile and a zero-filled ring (edge reads stay finite)
    tile_z_setup<VEL>(S, g, ts, z0, box);
    {
        const int total = LEAD + STAGES * cap + SLACK;
        for (int i = threadIdx.x; i < total; i += blockDim.x) ring[i] = TT(0.f);
    }
    TB* tab = reinterpret_cast<TB*>(smem_raw + mig_static_bytes() + mig_ring_bytes(g));
    float2* srcc = reinterpret_cast<float2*>(smem_raw + mig_static_bytes() + mig_ring_bytes(g) + table_bytes(g));
    if constexpr (VEL == VK_TABLE) {
        const uint4* src = reinterpret_cast<const uint4*>(g.table);
        uint4* dst = reinterpret_cast<uint4*>(tab);
        const int n16 = (int)(table_bytes(g) / 16);
        for (int i = threadIdx.x; i < n16; i += blockDim.x) dst[i] = src[i];
    }
    __syncthreads();
    if (s_abort) return;
    if (threadIdx.x >= CONSUMERS) {
        mig_producer<VEL, TT, WGT>(S, data, cap, g, tr, traces, bin, box, wc, 0, (int)blockIdx.x,
                                   ts.seq ? ts.seq - 1 : (int)blockIdx.z, ts.split);
    } else if constexpr (MODE == 0) {
        mig_consumer<VEL, WGT, FAST, TT, LPT, TB>(S, data, g, ts, x0, y0, z0, box, bin, image + split_offset(g, blockIdx.z),
                                                  wc, tab, srcc, cap, 0);
    } else {
        vg_consumer<VEL, WGT, FAST, TT, LPT>(S, data, g, ts, x0, y0, z0, box, bin, image, partial, wc, srcc, cap);
    }
}

template <int VEL, int WGT, bool FAST, typename TT, int LPT, typename TB = float>
__global__ void __launch_bounds__(THREADS, 2)
    k_migrate(GeomParams g, TileShape ts, TraceSet tr, const TT* __restrict__ traces,
              float* __restrict__ image, int cap, WaitCfg wc)
{
    kernel_body<VEL, WGT, FAST, TT, LPT, 0, TB>(g, ts, tr, traces, image, cap, wc, nullptr);
}

template <int VEL, int WGT, bool FAST, typename TT, int LPT>
__global__ void __launch_bounds__(THREADS, 2)
    k_vgrad(GeomParams g, TileShape ts, TraceSet tr, const TT* __restrict__ traces,
            const float* __restrict__ image, int cap, WaitCfg wc, double* __restrict__ partial)
{
    kernel_body<VEL, WGT, FAST, TT, LPT, 1>(g, ts, tr, traces, const_cast<float*>(image), cap, wc, partial);
}

// ------------------------------------------------------------------ launch (per trace type)
template <int VEL, int WGT, bool FAST, typename TT>
static cudaError_t launch_migrate_t(const GeomParams& g, const TileShape& t, const TraceSet& tr,
                                   const void* traces, float* image, const WaitCfg& w, cudaStream_t s)
{
    const size_t smem = mig_smem_bytes(g);
    const dim3 grid((unsigned)(t.tiles_x * t.tiles_y * t.tiles_z), (unsigned)g.n_bins, (unsigned)(t.seq ? 1 : t.split));
    auto go = [&](auto kern) -> cudaError_t {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        kern<<<grid, THREADS, smem, s>>>(g, t, tr, static_cast<const TT*>(traces), image, mig_cap(g), w);
        return cudaGetLastError();
    };
    if constexpr (VEL == VK_LINEAR) {
        return with_lg<FAST>(g.lg_terms,
                             [&](auto L) { return go(k_migrate<VEL, WGT, FAST, TT, decltype(L)::value>); });
    } else if constexpr (VEL == VK_GRID) {
        // the LPT slot carries the tables' depth-node stride M
        switch (g.tm) {
            case 1: return go(k_migrate<VEL, WGT, FAST, TT, 1>);
            case 2: return go(k_migrate<VEL, WGT, FAST, TT, 2>);
            case 4: return go(k_migrate<VEL, WGT, FAST, TT, 4>);
            default: return cudaErrorInvalidValue;
        }
    } else if constexpr (VEL == VK_TABLE) {
        // the LPT slot carries the table's depth-node stride M
        auto tb = [&](auto M) -> cudaError_t {
            constexpr int m = decltype(M)::value;
            if (g.tdt == KH_F16) return go(k_migrate<VEL, WGT, FAST, TT, m, __half>);
            if (g.tdt == KH_U16) return go(k_migrate<VEL, WGT, FAST, TT, m, unsigned short>);
            return go(k_migrate<VEL, WGT, FAST, TT, m, float>);
        };
        switch (g.tm) {
            case 1: return tb(std::integral_constant<int, 1>());
            case 2: return tb(std::integral_constant<int, 2>());
            case 4: return tb(std::integral_constant<int, 4>());
            default: return cudaErrorInvalidValue;
        }
    } else {
        return go(k_migrate<VEL, WGT, FAST, TT, LP_SHORT>);
    }
}

// Operator anti-aliasing (g.aa_c > 0): the kernels compiled with the W_AA bit, instantiated in
// translation units of their own (kh_migrate_aa_<type>.cu) so that they build beside the others;
// constant velocity for every trace type, v0 + k z for FP32 traces (the plan refuses the others).
template <typename TT>
cudaError_t launch_migrate_aa_t(const GeomParams& g, const TileShape& t, const TraceSet& tr, const void* traces,
                                float* image, int vel, int fast, const WaitCfg& w, cudaStream_t s)
{
    if (vel == VK_LINEAR) {   // v0 + k z: FP32 traces only (the plan refuses the others)
        if constexpr (std::is_same<TT, float>::value || std::is_same<TT, SamplePair>::value) {
            switch (g.weight * 2 + (fast ? 1 : 0)) {
                case 0: return launch_migrate_t<VK_LINEAR, W_AA | 0, false, TT>(g, t, tr, traces, image, w, s);
                case 1: return launch_migrate_t<VK_LINEAR, W_AA | 0, true, TT>(g, t, tr, traces, image, w, s);
                case 2: return launch_migrate_t<VK_LINEAR, W_AA | 1, false, TT>(g, t, tr, traces, image, w, s);
                case 3: return launch_migrate_t<VK_LINEAR, W_AA | 1, true, TT>(g, t, tr, traces, image, w, s);
                default: return cudaErrorInvalidValue;
            }
        } else {
            return cudaErrorInvalidValue;
        }
    }
    if (vel != VK_CONST) return cudaErrorInvalidValue;
    switch (g.weight * 2 + (fast ? 1 : 0)) {
        case 0: return launch_migrate_t<VK_CONST, W_AA | 0, false, TT>(g, t, tr, traces, image, w, s);
        case 1: return launch_migrate_t<VK_CONST, W_AA | 0, true, TT>(g, t, tr, traces, image, w, s);
        case 2: return launch_migrate_t<VK_CONST, W_AA | 1, false, TT>(g, t, tr, traces, image, w, s);
        case 3: return launch_migrate_t<VK_CONST, W_AA | 1, true, TT>(g, t, tr, traces, image, w, s);
        case 4: return launch_migrate_t<VK_CONST, W_AA | 2, false, TT>(g, t, tr, traces, image, w, s);
        case 5: return launch_migrate_t<VK_CONST, W_AA | 2, true, TT>(g, t, tr, traces, image, w, s);
        default: return cudaErrorInvalidValue;
    }
}

// Radial tables (fast math only).
template <typename TT>
cudaError_t launch_migrate_table_t(const GeomParams& g, const TileShape& t, const TraceSet& tr, const void* traces,
                                   float* image, const WaitCfg& w, cudaStream_t s)
{
    return g.weight == 1 ? launch_migrate_t<VK_TABLE, 1, true, TT>(g, t, tr, traces, image, w, s)
                         : launch_migrate_t<VK_TABLE, 0, true, TT>(g, t, tr, traces, image, w, s);
}

template <typename TT>
cudaError_t launch_migrate_dtype(const GeomParams& g, const TileShape& t, const TraceSet& tr, const void* traces,
                                 float* image, int vel, int fast, const WaitCfg& w, cudaStream_t s)
{
    if (g.weight == KH_W_TRUE_AMP) {   // constant velocity only (the plan refuses the others)
        if (vel != VK_CONST) return cudaErrorInvalidValue;
        return fast ? launch_migrate_t<VK_CONST, 2, true, TT>(g, t, tr, traces, image, w, s)
                    : launch_migrate_t<VK_CONST, 2, false, TT>(g, t, tr, traces, image, w, s);
    }
    const int key = vel * 4 + g.weight * 2 + (fast ? 1 : 0);
    switch (key) {
        case 0: return launch_migrate_t<VK_CONST, 0, false, TT>(g, t, tr, traces, image, w, s);
        case 1: return launch_migrate_t<VK_CONST, 0, true, TT>(g, t, tr, traces, image, w, s);
        case 2: return launch_migrate_t<VK_CONST, 1, false, TT>(g, t, tr, traces, image, w, s);
        case 3: return launch_migrate_t<VK_CONST, 1, true, TT>(g, t, tr, traces, image, w, s);
        case 4: return launch_migrate_t<VK_LINEAR, 0, false, TT>(g, t, tr, traces, image, w, s);
        case 5: return launch_migrate_t<VK_LINEAR, 0, true, TT>(g, t, tr, traces, image, w, s);
        case 6: return launch_migrate_t<VK_LINEAR, 1, false, TT>(g, t, tr, traces, image, w, s);
        case 7: return launch_migrate_t<VK_LINEAR, 1, true, TT>(g, t, tr, traces, image, w, s);
        case 8:
        case 9: return launch_migrate_t<VK_TABLE, 0, true, TT>(g, t, tr, traces, image, w, s);
        case 10:
        case 11: return launch_migrate_t<VK_TABLE, 1, true, TT>(g, t, tr, traces, image, w, s);
        case 12: return launch_migrate_t<VK_PSTM, 0, false, TT>(g, t, tr, traces, image, w, s);
        case 13: return launch_migrate_t<VK_PSTM, 0, true, TT>(g, t, tr, traces, image, w, s);
        case 14: return launch_migrate_t<VK_PSTM, 1, false, TT>(g, t, tr, traces, image, w, s);
        case 15: return launch_migrate_t<VK_PSTM, 1, true, TT>(g, t, tr, traces, image, w, s);
        case 16:
        case 17: return launch_migrate_t<VK_GRID, 0, true, TT>(g, t, tr, traces, image, w, s);
        case 18:
        case 19: return launch_migrate_t<VK_GRID, 1, true, TT>(g, t, tr, traces, image, w, s);
        default: return cudaErrorInvalidValue;
    }
}

// Gradient kernel (FP32 traces, analytic traveltimes only).
template <int VEL, int WGT, bool FAST>
static cudaError_t launch_vgrad_t(const GeomParams& g, const TileShape& t, const TraceSet& tr,
                                 const float* traces, const float* image, const WaitCfg& w, double* partial,
                                 cudaStream_t s)
{
    const size_t smem = mig_smem_bytes(g);
    const dim3 grid((unsigned)(t.tiles_x * t.tiles_y * t.tiles_z), (unsigned)g.n_bins, (unsigned)t.split);
    auto go = [&](auto kern) -> cudaError_t {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        kern<<<grid, THREADS, smem, s>>>(g, t, tr, traces, image, mig_cap(g), w, partial);
        return cudaGetLastError();
    };
    if constexpr (VEL == VK_LINEAR)
        return with_lg<FAST>(g.lg_terms,
                             [&](auto L) { return go(k_vgrad<VEL, WGT, FAST, float, decltype(L)::value>); });
    else
        return go(k_vgrad<VEL, WGT, FAST, float, LP_SHORT>);
}

// ------------------------------------------------------------------ batched persistent launch
// One CTA per (SM, resident slot) loops over a work list of (job, tile, bin) items, longest
// first, taking the next item from one global counter (a scheduler index, never image data).
// Each item is the tile computation of k_migrate with the job's own geometry, tile shape,
// headers, traces and image; the mbarrier ring and its phases persist across items.  All jobs
// of one launch share the ln(1 + rho) fit length LPT (the host launches the jobs of each fit
// length separately).  A wait that ran out anywhere in the launch (status word) stops
// every CTA at its next item.
template <int VEL, int WGT, bool FAST, typename TT, int LPT>
__global__ void __launch_bounds__(THREADS, 2)
    k_migrate_batched(const BatchJob* __restrict__ jobs, const int4* __restrict__ items, int n_items,
                      int* __restrict__ next, GeomParams g_ring, WaitCfg wc)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    MigSmem& S = *reinterpret_cast<MigSmem*>(smem_raw);
    TT* ring = reinterpret_cast<TT*>(smem_raw + mig_static_bytes());
    TT* data = ring + LEAD;
    float2* srcc = reinterpret_cast<float2*>(smem_raw + mig_static_bytes() + mig_ring_bytes(g_ring));
    __shared__ int s_item;
    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&S.full[s], 1);
            mbar_init(&S.empty[s], CONSUMER_WARPS);
        }
        S.zero[0] = S.zero[1] = S.zero[2] = S.zero[3] = 0.f;
        fence_barrier_init();
    }
    const int cap = mig_cap(g_ring);
    for (int i = threadIdx.x; i < LEAD + STAGES * cap + SLACK; i += blockDim.x) ring[i] = TT(0.f);
    int n = 0;   // stages filled (producer warp) or consumed (consumer warps) so far
    while (true) {
        __syncthreads();   // the previous item's per-z constants and s_item are no longer read
        if (threadIdx.x == 0) {
            const int bad = *reinterpret_cast<const volatile int*>(wc.status);
            s_item = bad ? n_items : atomicAdd(next, 1);
        }
        __syncthreads();
        const int it = s_item;
        if (it >= n_items) break;
        const int4 w = items[it];
        const GeomParams g = jobs[w.x].g;
        TileShape ts = jobs[w.x].ts;
        if (ts.seq) ts.seq = w.w + 1;
        const TraceSet tr = jobs[w.x].tr;
        int t = w.y;
        const int tzi = t % ts.tiles_z;
        t /= ts.tiles_z;
        const int txi = t % ts.tiles_x, tyi = t / ts.tiles_x;
        const int x0 = txi * ts.cx, y0 = tyi * ts.cy, z0 = tzi * ts.cz * NZ;
        const int bin = w.z;
        const TileBox box = tile_box(g, x0, y0, z0, ts.cx, ts.cy, ts.cz * NZ);
        tile_z_setup<VEL>(S, g, ts, z0, box);
        if (threadIdx.x == 0) tile_cells(S.row, tr, box);
        __syncthreads();
        if (threadIdx.x >= CONSUMERS) {
            n = mig_producer<VEL, TT>(S, data, cap, g, tr, static_cast<const TT*>(jobs[w.x].traces),
                                      bin, box, wc, n, 0, w.w, ts.split);
        } else {
            n = mig_consumer<VEL, WGT, FAST, TT, LPT, float>(S, data, g, ts, x0, y0, z0, box, bin,
                                                             jobs[w.x].image + (ts.seq ? 0 : split_offset(g, w.w)), wc,
                                                             nullptr, srcc, cap, n);
        }
    }
}

template <int VEL, int WGT, bool FAST, typename TT>
static cudaError_t launch_batched_t(const GeomParams& gm, const BatchJob* jobs, const int4* items,
                                   int n_items, int* next, int lg_terms, const WaitCfg& w, int ctas,
                                   int* ctas_out, cudaStream_t s)
{
    const size_t smem = mig_smem_bytes(gm);
    auto go = [&](auto kern) -> cudaError_t {
        cudaError_t e;
        if (ctas <= 0) {   // set-up only: shared-memory attribute and the occupancy-sized grid
            int dev = 0, nsm = 0, occ = 0;
            if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) !=
                cudaSuccess)
                return e;
            if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
            if ((e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
            if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, THREADS, smem)) != cudaSuccess)
                return e;
            int c = nsm * (occ > 0 ? occ : 1);
            if (c > n_items) c = n_items;
            if (ctas_out) *ctas_out = c;
            return cudaSuccess;
        }
        kern<<<ctas, THREADS, smem, s>>>(jobs, items, n_items, next, gm, w);
        return cudaGetLastError();
    };
    if constexpr (VEL == VK_LINEAR)
        return with_lg<FAST>(lg_terms,
                             [&](auto L) { return go(k_migrate_batched<VEL, WGT, FAST, TT, decltype(L)::value>); });
    else
        return go(k_migrate_batched<VEL, WGT, FAST, TT, LP_SHORT>);
}

template <typename TT>
cudaError_t launch_batched_dtype(const GeomParams& gm, const BatchJob* jobs, const int4* items, int n_items,
                                 int* next, int vel, int weight, int fast, int lg_terms, const WaitCfg& w,
                                 int ctas, int* ctas_out, cudaStream_t s)
{
    const int key = vel * 4 + weight * 2 + (fast ? 1 : 0);
    switch (key) {
        case 0: return launch_batched_t<VK_CONST, 0, false, TT>(gm, jobs, items, n_items, next, lg_terms, w, ctas, ctas_out, s);
        case 1: return launch_batched_t<VK_CONST, 0, true, TT>(gm, jobs, items, n_items, next, lg_terms, w, ctas, ctas_out, s);
        case 2: return launch_batched_t<VK_CONST, 1, false, TT>(gm, jobs, items, n_items, next, lg_terms, w, ctas, ctas_out, s);
        case 3: return launch_batched_t<VK_CONST, 1, true, TT>(gm, jobs, items, n_items, next, lg_terms, w, ctas, ctas_out, s);
        case 4: return launch_batched_t<VK_LINEAR, 0, false, TT>(gm, jobs, items, n_items, next, lg_terms, w, ctas, ctas_out, s);
        case 5: return launch_batched_t<VK_LINEAR, 0, true, TT>(gm, jobs, items, n_items, next, lg_terms, w, ctas, ctas_out, s);
        case 6: return launch_batched_t<VK_LINEAR, 1, false, TT>(gm, jobs, items, n_items, next, lg_terms, w, ctas, ctas_out, s);
        case 7: return launch_batched_t<VK_LINEAR, 1, true, TT>(gm, jobs, items, n_items, next, lg_terms, w, ctas, ctas_out, s);
        default: return cudaErrorInvalidValue;
    }
}


}  // namespace kh
