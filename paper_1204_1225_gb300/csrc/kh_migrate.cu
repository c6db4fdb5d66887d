// Migration, batched-migration and velocity-gradient launches: dispatch on the trace type to
// the per-type translation units (kh_migrate_<type>.cu, kh_migrate_aa_<type>.cu with operator
// anti-aliasing, kh_batched_<type>.cu), the gradient
// kernels (FP32 traces only, instantiated here) and the gradient's final sum.
#include "kh_migrate_impl.cuh"

namespace kh {

#define KH_MIGRATE_DECL(name)                                                                            \
    cudaError_t name(const GeomParams&, const TileShape&, const TraceSet&, const void*, float*, int, int,     \
                     const WaitCfg&, cudaStream_t);
KH_MIGRATE_DECL(launch_migrate_f32)
KH_MIGRATE_DECL(launch_migrate_pair)
KH_MIGRATE_DECL(launch_migrate_f16)
KH_MIGRATE_DECL(launch_migrate_bf16)
KH_MIGRATE_DECL(launch_migrate_pair_table)
KH_MIGRATE_DECL(launch_migrate_aa_f32)
KH_MIGRATE_DECL(launch_migrate_aa_pair)
KH_MIGRATE_DECL(launch_migrate_aa_f16)
KH_MIGRATE_DECL(launch_migrate_aa_bf16)
#undef KH_MIGRATE_DECL

#define KH_BATCHED_DECL(name)                                                                            \
    cudaError_t name(const GeomParams&, const BatchJob*, const int4*, int, int*, int, int, int, int,          \
                     const WaitCfg&, int, int*, cudaStream_t);
KH_BATCHED_DECL(launch_batched_f32)
KH_BATCHED_DECL(launch_batched_pair)
KH_BATCHED_DECL(launch_batched_f16)
KH_BATCHED_DECL(launch_batched_bf16)
#undef KH_BATCHED_DECL

size_t migrate_smem_bytes(const GeomParams& g) { return mig_smem_bytes(g); }
bool migrate_fits_twice(const GeomParams& g) { return mig_smem_bytes(g) <= CTA_SMEM_BUDGET; }

cudaError_t launch_migrate_batched(const GeomParams& gm, const BatchJob* jobs, const int4* items, int n_items,
                                   int* next, int vel_kind, int weight, int fast, int lg_terms,
                                   int trace_dtype, const WaitCfg& w, int ctas, int* ctas_out,
                                   cudaStream_t s)
{
    switch (trace_dtype) {
        case KH_F32:
            if (gm.pairs)
                return launch_batched_pair(gm, jobs, items, n_items, next, vel_kind, weight, fast, lg_terms, w, ctas,
                                           ctas_out, s);
            return launch_batched_f32(gm, jobs, items, n_items, next, vel_kind, weight, fast, lg_terms, w, ctas,
                                      ctas_out, s);
        case KH_F16:
            return launch_batched_f16(gm, jobs, items, n_items, next, vel_kind, weight, fast, lg_terms, w, ctas,
                                      ctas_out, s);
        case KH_BF16:
            return launch_batched_bf16(gm, jobs, items, n_items, next, vel_kind, weight, fast, lg_terms, w, ctas,
                                       ctas_out, s);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_migrate(const GeomParams& g, const TileShape& t, const TraceSet& tr,
                           const void* traces, float* image, int vel_kind, int fast_math,
                           const WaitCfg& w, cudaStream_t s)
{
    if (t.cz > MAX_ZG) return cudaErrorInvalidValue;
    if (g.pstm) vel_kind = VK_PSTM;   // time migration has kernels of its own
    if (g.aa_c > 0.f) {   // operator anti-aliasing has kernels of its own
        switch (g.tdtype) {
            case KH_F32:
                return g.pairs ? launch_migrate_aa_pair(g, t, tr, traces, image, vel_kind, fast_math, w, s)
                               : launch_migrate_aa_f32(g, t, tr, traces, image, vel_kind, fast_math, w, s);
            case KH_F16: return launch_migrate_aa_f16(g, t, tr, traces, image, vel_kind, fast_math, w, s);
            case KH_BF16: return launch_migrate_aa_bf16(g, t, tr, traces, image, vel_kind, fast_math, w, s);
            default: return cudaErrorInvalidValue;
        }
    }
    if (g.pairs && vel_kind == VK_TABLE)
        return launch_migrate_pair_table(g, t, tr, traces, image, vel_kind, fast_math, w, s);
    switch (g.tdtype) {
        case KH_F32:
            return g.pairs ? launch_migrate_pair(g, t, tr, traces, image, vel_kind, fast_math, w, s)
                           : launch_migrate_f32(g, t, tr, traces, image, vel_kind, fast_math, w, s);
        case KH_F16: return launch_migrate_f16(g, t, tr, traces, image, vel_kind, fast_math, w, s);
        case KH_BF16: return launch_migrate_bf16(g, t, tr, traces, image, vel_kind, fast_math, w, s);
        default: return cudaErrorInvalidValue;
    }
}

// Splitting pays while the CTAs (a tile and a bin each) leave SMs idle: below two waves of the 304 that
// run at once.  Time model, in units of one staged trace of a CTA (about 1.2 us): the waves times a
// part's traces and a CTA's set-up (8), plus the partial images' write and read and the summing
// launch; parts keep at least 16 traces and their images 512 MB, and a split has to promise a tenth (a
// batch's work list fills the SMs without it and pays for the partial images).  Measured, kernel and sum:
// 128 x 128 points, 1024 traces, 8 bins (32 CTAs, 8 parts) 85 -> 32 us; 128 x 100, 4608 traces, 4 bins (16 CTAs,
// 19 parts) 1855 -> 136 us, its gradient 2054 -> 188 us; 160 x 120, 2400 traces, 8 bins (48 CTAs, 6 parts) 260
// -> 94 us; 512 x 400, 20 000 traces, 8 bins (448 CTAs, 1.5 waves, 2 parts) 4.65 -> 4.20 ms.
int split_of(const GeomParams& g, const TileShape& t, int ntr)
{
    constexpr int SLOTS = 2 * 152;
    const long long n = (long long)t.tiles_x * t.tiles_y * t.tiles_z * g.n_bins;
    if (n >= 2 * SLOTS) return 1;
    const double per = (double)ntr / g.n_bins;
    const double image = 4.0 * g.n_bins * g.ny * g.nx * (double)g.nz;
    int best = 1;
    double least = 1e300;
    for (int s = 1; s <= MAX_SPLIT && (s == 1 || (per >= 16.0 * s && image * s <= 512e6)); ++s) {
        const double waves = (double)((n * s + SLOTS - 1) / SLOTS);
        const double cost = waves * (per / s + 8.0) + (s > 1 ? 3.0 + s * image / 4e6 : 0.0);
        if (cost < (best == 1 ? 0.9 : 0.97) * least) {
            least = cost;
            best = s;
        }
    }
    return best;
}

// One thread four samples; the partial images are read once.
__global__ void __launch_bounds__(256) k_split_sum(const float* __restrict__ part, int split, long long n,
                                                   float* __restrict__ image)
{
    const long long step = 4LL * gridDim.x * blockDim.x;
    const bool vec = (n & 3) == 0 && (reinterpret_cast<uintptr_t>(image) & 15) == 0;
    for (long long i = 4 * (blockIdx.x * (long long)blockDim.x + threadIdx.x); i < n; i += step) {
        if (vec) {
            float4 s = *reinterpret_cast<const float4*>(part + i);
#pragma unroll 4
            for (int k = 1; k < split; ++k) {
                const float4 v = *reinterpret_cast<const float4*>(part + k * n + i);
                s.x += v.x;
                s.y += v.y;
                s.z += v.z;
                s.w += v.w;
            }
            *reinterpret_cast<float4*>(image + i) = s;
        } else {
            for (long long e = i; e < min(i + 4, n); ++e) {
                float s = part[e];
                for (int k = 1; k < split; ++k) s += part[k * n + e];
                image[e] = s;
            }
        }
    }
}

cudaError_t launch_split_sum(const float* partial, int split, long long n, float* image, cudaStream_t s)
{
    const long long blocks = (n + 1023) / 1024;
    k_split_sum<<<(unsigned)(blocks < 1 ? 1 : blocks > 152 * 16 ? 152 * 16 : blocks), 256, 0, s>>>(partial, split, n, image);
    return cudaGetLastError();
}

static cudaError_t launch_vgrad_impl(const GeomParams& g, const TileShape& t, const TraceSet& tr,
                                     const float* traces, const float* image, int vel, int fast, const WaitCfg& w,
                                     double* partial, cudaStream_t s)
{
    const int key = vel * 4 + g.weight * 2 + (fast ? 1 : 0);
    switch (key) {
        case 0: return launch_vgrad_t<VK_CONST, 0, false>(g, t, tr, traces, image, w, partial, s);
        case 1: return launch_vgrad_t<VK_CONST, 0, true>(g, t, tr, traces, image, w, partial, s);
        case 2: return launch_vgrad_t<VK_CONST, 1, false>(g, t, tr, traces, image, w, partial, s);
        case 3: return launch_vgrad_t<VK_CONST, 1, true>(g, t, tr, traces, image, w, partial, s);
        case 4: return launch_vgrad_t<VK_LINEAR, 0, false>(g, t, tr, traces, image, w, partial, s);
        case 5: return launch_vgrad_t<VK_LINEAR, 0, true>(g, t, tr, traces, image, w, partial, s);
        case 6: return launch_vgrad_t<VK_LINEAR, 1, false>(g, t, tr, traces, image, w, partial, s);
        case 7: return launch_vgrad_t<VK_LINEAR, 1, true>(g, t, tr, traces, image, w, partial, s);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_vgrad(const GeomParams& g, const TileShape& t, const TraceSet& tr,
                         const void* traces, const float* image, int vel_kind, int fast_math,
                         const WaitCfg& w, double* partial, cudaStream_t s)
{
    if (t.cz > MAX_ZG || !partial) return cudaErrorInvalidValue;
    if (g.tdtype != KH_F32 || vel_kind == VK_TABLE || g.weight == KH_W_TRUE_AMP) return cudaErrorInvalidValue;
    return launch_vgrad_impl(g, t, tr, static_cast<const float*>(traces), image, vel_kind, fast_math, w, partial,
                             s);
}

// out[0..1] = (sum of the per-warp partials, in index order) / dt: one CTA, fixed order.
__global__ void k_vgrad_reduce(const double* __restrict__ partial, long long n, double inv_dt,
                               double* __restrict__ out)
{
    __shared__ double s0[256], s1[256];
    double a = 0.0, b = 0.0;
    for (long long i = threadIdx.x; i < n; i += blockDim.x) {
        a += partial[2 * i];
        b += partial[2 * i + 1];
    }
    s0[threadIdx.x] = a;
    s1[threadIdx.x] = b;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) {
            s0[threadIdx.x] += s0[threadIdx.x + w];
            s1[threadIdx.x] += s1[threadIdx.x + w];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        out[0] = s0[0] * inv_dt;
        out[1] = s1[0] * inv_dt;
    }
}

cudaError_t launch_vgrad_reduce(const double* partial, long long n, double inv_dt, double* out,
                                cudaStream_t s)
{
    k_vgrad_reduce<<<1, 256, 0, s>>>(partial, n, inv_dt, out);
    return cudaGetLastError();
}

}  // namespace kh
