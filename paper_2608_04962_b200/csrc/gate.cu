// Reliability side of the hidden-state correction (Sec. 3.4 "Reliability from delayed alignment", Eq.
// "reliability-score", the indicator of Eq. "reflex-correction"; App. "Implementation details", paragraph
// "Reflex configuration"): normalised random-projection sketches, realised alignments, exact online sample
// moments per (trajectory, horizon) slot, the conservative score and the gate that yields the correction ratio.
// Small, latency-bound kernels: a few thousand records and slots per call.
#include <math.h>

#include <algorithm>

#include "common.cuh"

namespace specroll {

namespace gt {
constexpr int SK_THREADS = 256;
constexpr int SK_WARPS = SK_THREADS / 32;
constexpr int MAX_RANK = 32;
constexpr int SK_CLUSTER = 4;   // CTAs that share the columns of their records
constexpr int SK_SMEM = 208 * 1024;
constexpr int GATE_THREADS = 128;
constexpr int GATE_BATCH = 4 * GATE_THREADS;
}  // namespace gt

// y = Pi x (rank dot products of length d), then y / ||y||; d % 4 == 0 and 16-byte aligned rows.
// Pi is a few hundred KB that every record meets: with a CTA per record the kernel was bound by bringing it from L2 once
// per record (512 records, d 3584, rank 24: 17-22 us).  A cluster of four CTAs takes RECS records, each CTA a quarter of
// the columns: it asks for its part of Pi and of the records in one go (asynchronous copies, `cols` columns of four at a
// time), so there is one memory latency and not one per step of a loop; the partial dot products meet in distributed
// shared memory.  Within a CTA a warp has four records and every CS-th group of 32 columns: what the products read of shared
// memory is what bounds them then, and with one or two records per warp that was twice to three times as much
// (9.7 -> 9.0 us).
template <int RECS>
__global__ void __launch_bounds__(gt::SK_THREADS) sketch_kernel(int R, int d4, int rank, int cols, const float4 *__restrict__ X,
                                                                 const int32_t *__restrict__ rows,
                                                                 const float4 *__restrict__ Pi, float *__restrict__ sketch) {
    using namespace gt;
    constexpr int QUADS = RECS / 4, CS = SK_WARPS / QUADS;
    __shared__ float part[CS][RECS][MAX_RANK];
    extern __shared__ __align__(16) float4 sh_cols[];  // [rank + RECS][cols]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, cta = (int)cluster_ctarank();
    const int quad = warp % QUADS, cs = warp / QUADS;
    const int r0 = (blockIdx.x / SK_CLUSTER) * RECS;
    const int per = (d4 + SK_CLUSTER - 1) / SK_CLUSTER, c0 = min(d4, cta * per), c1 = min(d4, c0 + per);
    for (int e = threadIdx.x; e < CS * RECS * MAX_RANK; e += SK_THREADS) (&part[0][0][0])[e] = 0.f;
    pdl_wait();
    pdl_launch_dependents();
    for (int cb = c0; cb < c1; cb += cols) {
        const int n = min(cols, c1 - cb);
        __syncthreads();  // (part cleared; the columns before have been read)
        for (int i = warp; i < rank + RECS; i += SK_WARPS) {
            const int r = min(r0 + i - rank, R - 1);  // (beyond the last record: its copy, not written)
            const float4 *src = (i < rank ? Pi + (size_t)i * d4 : X + (size_t)(rows ? rows[r] : r) * d4) + cb;
            for (int c = lane; c < n; c += 32) cp_async16(smem_u32(sh_cols + (size_t)i * cols + c), src + c, true);
        }
        cp_async_commit();
        cp_async_wait<0>();
        __syncthreads();
        const float4 *x = sh_cols + (size_t)(rank + quad * 4) * cols;
        for (int i0 = 0; i0 < rank; i0 += 8) {  // eight ranks at a time: 32 independent sums
            float acc[32];
#pragma unroll
            for (int q = 0; q < 32; ++q) acc[q] = 0.f;
            for (int c = lane + 32 * cs; c < n; c += 32 * CS) {
                float4 xv[4];
#pragma unroll
                for (int v = 0; v < 4; ++v) xv[v] = x[v * cols + c];
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const float4 pv = sh_cols[(size_t)min(i0 + q, rank - 1) * cols + c];
#pragma unroll
                    for (int v = 0; v < 4; ++v)
                        acc[v * 8 + q] = fmaf(pv.x, xv[v].x, fmaf(pv.y, xv[v].y, fmaf(pv.z, xv[v].z, fmaf(pv.w, xv[v].w, acc[v * 8 + q]))));
                }
            }
            part[cs][quad * 4 + lane / 8][i0 + lane % 8] += warp_sum_many<5>(acc, lane);  // (a warp's own entries)
        }
    }
    cluster_sync_all();
    // records in turn over the cluster's warps
    for (int j = cta * SK_WARPS + warp; j < RECS && r0 + j < R; j += SK_CLUSTER * SK_WARPS) {
        float v = 0.f;
        if (lane < rank)
#pragma unroll
            for (int k = 0; k < SK_CLUSTER; ++k)
#pragma unroll
                for (int q = 0; q < CS; ++q) v += __uint_as_float(ld_dsmem_u32(&part[q][j][lane], k));
        const float nrm = sqrtf(warp_sum(v * v));
        if (lane < rank) sketch[(size_t)(r0 + j) * rank + lane] = nrm > 0.f ? v / nrm : 0.f;
    }
    cluster_sync_all();  // (a CTA's partial products stay until all have read them)
}

// The same for any d and alignment: a CTA per record, a warp takes the ranks warp, warp + 8, ... (four at most).
__global__ void __launch_bounds__(gt::SK_THREADS) sketch_any_kernel(int d, int rank, const float *__restrict__ X,
                                                                     const int32_t *__restrict__ rows,
                                                                     const float *__restrict__ Pi, float *__restrict__ sketch) {
    __shared__ float y[gt::MAX_RANK];
    constexpr int NW = gt::SK_WARPS, RPW = gt::MAX_RANK / NW;
    const int r = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    pdl_wait();
    pdl_launch_dependents();
    const float *x = X + (size_t)(rows ? rows[r] : r) * d;
    float acc[RPW];
#pragma unroll
    for (int q = 0; q < RPW; ++q) acc[q] = 0.f;
    for (int c = lane; c < d; c += 32) {
        const float xv = x[c];
#pragma unroll
        for (int q = 0; q < RPW; ++q) {
            const int i = warp + q * NW;
            if (i < rank) acc[q] = fmaf(Pi[(size_t)i * d + c], xv, acc[q]);
        }
    }
#pragma unroll
    for (int q = 0; q < RPW; ++q) {
        const float t = warp_sum(acc[q]);
        if (lane == 0 && warp + q * NW < rank) y[warp + q * NW] = t;
    }
    __syncthreads();
    if (warp == 0) {
        const float v = lane < rank ? y[lane] : 0.f;
        const float nrm = sqrtf(warp_sum(v * v));
        if (lane < rank) sketch[(size_t)r * rank + lane] = nrm > 0.f ? v / nrm : 0.f;
    }
}

struct GateArgs {
    const float *s, *xi;
    const int32_t *slot;
    const uint8_t *keep;
    int32_t *n, *n_fb;
    float *mean, *M2;
    const float *m;
    const int32_t *horizon, *n_align_min, *n_fb_min;
    const float *alpha_lo, *alpha_hi;
    float *a, *rel, *alpha;
    int R, S, d, rank, H;
    float z_delta, mem_eps;
};

// Realised alignment of record r, by a warp.
__device__ __forceinline__ float alignment(const GateArgs &g, int r, int lane) {
    const float sv = lane < g.rank ? g.s[(size_t)r * g.rank + lane] : 0.f;
    const float xv = lane < g.rank ? g.xi[(size_t)r * g.rank + lane] : 0.f;
    const float dot = warp_sum(sv * xv), ns = sqrtf(warp_sum(sv * sv)), nx = sqrtf(warp_sum(xv * xv));
    return (ns > 0.f && nx > 0.f) ? dot / (ns * nx) : 0.f;
}

// A CTA per slot: its records, in order, go into the running moments; then the score and the gate, with the RMS of the
// memory row.  Bound by latency: all threads look for the slot's records (512 at a time) and have the memory row's loads
// in flight meanwhile (a warp per slot took 14 us for 512 slots and records of d 3584).  A record's alignment is formed by
// the CTA of its slot, a warp per record (a kernel of its own in front of this one cost its launch and round trips).
__global__ void __launch_bounds__(gt::GATE_THREADS) gate_kernel(GateArgs g) {
    using namespace gt;
    __shared__ int hit[GATE_BATCH];
    __shared__ float val[GATE_BATCH];
    __shared__ int lost[GATE_BATCH];
    __shared__ int n_hit, n_lost;
    __shared__ float red[GATE_THREADS / 32];
    const int j = blockIdx.x, tid = threadIdx.x, lane = tid & 31;
    pdl_wait();
    pdl_launch_dependents();
    if (tid == 0) n_hit = n_lost = 0;
    int n = g.n[j], nfb = g.n_fb[j];
    float mean = g.mean[j], M2 = g.M2[j];
    float ss = 0.f;
    const float *mr = g.m + (size_t)j * g.d;
    if ((g.d % 4) == 0 && (reinterpret_cast<uintptr_t>(g.m) & 15u) == 0) {
        const float4 *m4 = reinterpret_cast<const float4 *>(mr);
        float s4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 8
        for (int c = tid; c < (g.d >> 2); c += GATE_THREADS) {
            const float4 v = m4[c];
            s4[0] = fmaf(v.x, v.x, s4[0]);
            s4[1] = fmaf(v.y, v.y, s4[1]);
            s4[2] = fmaf(v.z, v.z, s4[2]);
            s4[3] = fmaf(v.w, v.w, s4[3]);
        }
        ss = (s4[0] + s4[1]) + (s4[2] + s4[3]);
    } else {
        for (int c = tid; c < g.d; c += GATE_THREADS) ss = fmaf(mr[c], mr[c], ss);
    }
    __syncthreads();
    for (int r0 = 0; r0 < g.R; r0 += GATE_BATCH) {
        int sl[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int r = r0 + q * GATE_THREADS + tid;
            sl[q] = r < g.R ? g.slot[r] : -1;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int r = r0 + q * GATE_THREADS + tid;
            // (a record of no slot of this call has an alignment all the same: the first CTA's)
            const bool stray = j == 0 && (sl[q] < 0 || sl[q] >= g.S);
            if (r < g.R && (sl[q] == j || stray)) {
                if (g.keep && !g.keep[r])
                    g.a[r] = __int_as_float(0x7fc00000);
                else if (stray)
                    lost[atomicAdd(&n_lost, 1)] = r;
                else
                    hit[atomicAdd(&n_hit, 1)] = r;
            }
        }
        __syncthreads();
        const int nh = n_hit, nl = n_lost;
        __syncthreads();  // (all have read them before the next records are counted)
        if (nh + nl == 0) continue;
        for (int e = tid >> 5; e < nl; e += GATE_THREADS / 32) {
            const float v = alignment(g, lost[e], lane);
            if (lane == 0) g.a[lost[e]] = v;
        }
        // in record order
        for (int e = tid >> 5; e < nh; e += GATE_THREADS / 32) {
            const int r = hit[e];
            int rk = 0;
            for (int f = lane; f < nh; f += 32) rk += hit[f] < r;
            rk = __reduce_add_sync(0xffffffffu, rk);
            const float v = alignment(g, r, lane);
            if (lane == 0) {
                val[rk] = v;
                g.a[r] = v;
            }
        }
        __syncthreads();
        if (tid == 0) {
            n_hit = n_lost = 0;
            for (int e = 0; e < nh; ++e) {
                n += 1;
                const float delta = val[e] - mean;
                mean += delta / (float)n;
                M2 += delta * (val[e] - mean);
                nfb += 1;
            }
        }
        __syncthreads();
    }
    ss = warp_sum(ss);
    if (lane == 0) red[tid >> 5] = ss;
    __syncthreads();
    if (tid == 0) {
        ss = (red[0] + red[1]) + (red[2] + red[3]);
        g.n[j] = n;
        g.n_fb[j] = nfb;
        g.mean[j] = mean;
        g.M2[j] = M2;
        const int h = g.horizon[j];
        float rel = -INFINITY;
        if (n >= 2) rel = mean - g.z_delta * sqrtf(M2 / (float)(n - 1)) / sqrtf((float)n);
        const bool open = h >= 0 && h < g.H && n >= g.n_align_min[h] && nfb >= g.n_fb_min[h] && rel > 0.f &&
                          sqrtf(ss / (float)g.d) > g.mem_eps;
        g.rel[j] = rel;
        g.alpha[j] = open ? g.alpha_lo[h] + (g.alpha_hi[h] - g.alpha_lo[h]) * fminf(rel, 1.f) : 0.f;
    }
}

}  // namespace specroll

using namespace specroll;

extern "C" int specroll_reflex_sketch(int32_t R, int32_t d, int32_t rank, const float *X, const int32_t *rows,
                                      const float *Pi, float *sketch, void *cuda_stream) {
    if (R < 0 || d < 1 || rank < 1 || rank > gt::MAX_RANK) return SPECROLL_EINVAL;
    if (R == 0) return SPECROLL_OK;
    if (!X || !Pi || !sketch) return SPECROLL_EINVAL;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    if ((d % 4) == 0 && aligned16(X) && aligned16(Pi)) {
        // sixteen records per cluster halve the reads of Pi; with few records, eight, for more CTAs
        const int per = R > 296 ? 16 : 8, cols_all = (d / 4 + gt::SK_CLUSTER - 1) / gt::SK_CLUSTER;
        const int cols = std::min(cols_all, gt::SK_SMEM / 16 / (rank + per));
        auto *const kern = per == 16 ? sketch_kernel<16> : sketch_kernel<8>;
        const int rc = device_setup(reinterpret_cast<const void *>(kern), gt::SK_SMEM, nullptr);
        if (rc != SPECROLL_OK) return rc;
        SR_CUDA_TRY(launch_clusters(true, gt::SK_CLUSTER, kern, dim3((unsigned)((R + per - 1) / per * gt::SK_CLUSTER)),
                                    dim3(gt::SK_THREADS), (size_t)(rank + per) * cols * 16, st, R, d / 4, rank, cols,
                                    reinterpret_cast<const float4 *>(X), rows, reinterpret_cast<const float4 *>(Pi), sketch));
        return SPECROLL_OK;
    }
    SR_CUDA_TRY(launch_dependent(true, sketch_any_kernel, dim3((unsigned)R), dim3(gt::SK_THREADS), 0, st, d, rank, X, rows, Pi, sketch));
    return SPECROLL_OK;
}

extern "C" int specroll_reflex_gate(const specroll_gate_desc *d, const float *s, const float *xi, const int32_t *slot,
                                    const uint8_t *keep, int32_t *n, float *mean, float *M2, int32_t *n_fb,
                                    const float *m, const int32_t *horizon, const int32_t *n_align_min,
                                    const int32_t *n_fb_min, const float *alpha_lo, const float *alpha_hi, float *a,
                                    float *rel, float *alpha, void *cuda_stream) {
    if (!d || d->R < 0 || d->S < 1 || d->d < 1 || d->rank < 1 || d->rank > gt::MAX_RANK || d->H < 1 ||
        !(d->z_delta >= 0.f) || !(d->mem_eps >= 0.f) || d->flags != 0)
        return SPECROLL_EINVAL;
    if (!n || !mean || !M2 || !n_fb || !m || !horizon || !n_align_min || !n_fb_min || !alpha_lo || !alpha_hi || !rel ||
        !alpha)
        return SPECROLL_EINVAL;
    // the alignments are needed by the second kernel: without the caller's array there is nowhere to keep them
    if (d->R > 0 && (!s || !xi || !slot || !a)) return SPECROLL_EINVAL;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    GateArgs g;
    g.s = s;
    g.xi = xi;
    g.slot = slot;
    g.keep = keep;
    g.n = n;
    g.n_fb = n_fb;
    g.mean = mean;
    g.M2 = M2;
    g.m = m;
    g.horizon = horizon;
    g.n_align_min = n_align_min;
    g.n_fb_min = n_fb_min;
    g.alpha_lo = alpha_lo;
    g.alpha_hi = alpha_hi;
    g.a = a;
    g.rel = rel;
    g.alpha = alpha;
    g.R = d->R;
    g.S = d->S;
    g.d = d->d;
    g.rank = d->rank;
    g.H = d->H;
    g.z_delta = d->z_delta;
    g.mem_eps = d->mem_eps;
    SR_CUDA_TRY(launch_dependent(true, gate_kernel, dim3((unsigned)d->S), dim3(gt::GATE_THREADS), 0, st, g));
    return SPECROLL_OK;
}
