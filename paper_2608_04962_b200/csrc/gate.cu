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
constexpr int GATE_RECS_LOG = 3;            // a warp forms the alignments of eight records at once
// Up to so many records the gate forms their alignments itself, beyond it a kernel in front spreads them over the GPU.  A call, us
// (one launch less for the host as well; in a graph 512 of 512 slots 7.8 -> 7.0, 1024 of 16 13.7 -> 14.7, 64 of one 10.7 -> 12.3), in front -> itself (d 3584, rank 24): 512 records, one in each of 512 slots 14.9 -> 12.2, all in one 49 -> 43, of no slot 14.8 -> 12.2;
// 1024 of 1024 slots 14.9 -> 12.3, of 16 slots 15.0 -> 14.5; 640 of one slot 57 -> 53, 700 of five 18.6 -> 19.9, 512 of no slot in a
// call of one slot 14.5 -> 16.6.  Beyond: 4096 records of 16 slots 33.5 -> 35.0, of 512 slots 14.9 -> 18.6, one in each of 4096 24.7 -> 37.
constexpr int GATE_FEW = 8 * GATE_THREADS;
}  // namespace gt

// y = Pi x (rank dot products of length d), then y / ||y||; d % 4 == 0 and 16-byte aligned rows.
// Pi is a few hundred KB that every record meets: with a CTA per record the kernel was bound by bringing it from L2 once
// per record (512 records, d 3584, rank 24: 17-22 us).  A cluster of four CTAs takes RECS records, each CTA a quarter of
// the columns: it asks for its part of Pi and of the records in one go (asynchronous copies, `cols` columns of four at a
// time), so there is one memory latency and not one per step of a loop; the partial dot products meet in distributed
// shared memory.  Within a CTA a warp has VPW records and every CS-th group of 32 columns: where the columns are many, what the
// products read of shared memory bounds them, and that is the less the more records a warp has.
template <int RECS, int VPW>
__global__ void __launch_bounds__(gt::SK_THREADS) sketch_kernel(int R, int d4, int rank, int cols, const float4 *__restrict__ X,
                                                                 const int32_t *__restrict__ rows,
                                                                 const float4 *__restrict__ Pi, float *__restrict__ sketch) {
    using namespace gt;
    constexpr int GROUPS = RECS / VPW, CS = SK_WARPS / GROUPS, L = VPW == 4 ? 5 : VPW == 2 ? 4 : 3;
    __shared__ float part[CS][RECS][MAX_RANK];
    extern __shared__ __align__(16) float4 sh_cols[];  // [rank + RECS][cols]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, cta = (int)cluster_ctarank();
    const int grp = warp % GROUPS, cs = warp / GROUPS;
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
        const float4 *x = sh_cols + (size_t)(rank + grp * VPW) * cols;
        for (int i0 = 0; i0 < rank; i0 += 8) {  // eight ranks at a time: 8 VPW independent sums
            float acc[VPW * 8];
#pragma unroll
            for (int q = 0; q < VPW * 8; ++q) acc[q] = 0.f;
            for (int c = lane + 32 * cs; c < n; c += 32 * CS) {
                float4 xv[VPW];
#pragma unroll
                for (int v = 0; v < VPW; ++v) xv[v] = x[v * cols + c];
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const float4 pv = sh_cols[(size_t)min(i0 + q, rank - 1) * cols + c];
#pragma unroll
                    for (int v = 0; v < VPW; ++v)
                        acc[v * 8 + q] = fmaf(pv.x, xv[v].x, fmaf(pv.y, xv[v].y, fmaf(pv.z, xv[v].z, fmaf(pv.w, xv[v].w, acc[v * 8 + q]))));
                }
            }
            const float t = warp_sum_many<L>(acc, lane);
            const int e = lane >> (5 - L);
            if ((lane & ((1 << (5 - L)) - 1)) == 0) part[cs][grp * VPW + e / 8][i0 + e % 8] += t;  // (a warp's own entries)
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

// Realised alignments of the n records of list (the warp's own) to val (may be null) and g.a, by a warp.  The loads of 2^L records
// are in flight together; a sum is formed by the additions of warp_sum.
template <int L>
__device__ __forceinline__ void alignments(const GateArgs &g, const int *list, int n, float *val, int lane) {
    constexpr int RECS = 1 << L, LANES = 32 / RECS;
    for (int e0 = 0; e0 < n; e0 += RECS) {
        float dot[RECS], ns[RECS], nx[RECS];
#pragma unroll
        for (int q = 0; q < RECS; ++q) {
            const bool in = e0 + q < n && lane < g.rank;
            const size_t at = in ? (size_t)list[e0 + q] * g.rank + lane : 0;
            ns[q] = in ? g.s[at] : 0.f;
            nx[q] = in ? g.xi[at] : 0.f;
        }
#pragma unroll
        for (int q = 0; q < RECS; ++q) {
            dot[q] = ns[q] * nx[q];
            ns[q] *= ns[q];
            nx[q] *= nx[q];
        }
        const float d = warp_sum_many<L>(dot, lane), s = sqrtf(warp_sum_many<L>(ns, lane)), x = sqrtf(warp_sum_many<L>(nx, lane));
        const int e = e0 + lane / LANES;
        if (lane % LANES == 0 && e < n) {
            const float v = (s > 0.f && x > 0.f) ? d / (s * x) : 0.f;
            if (val) val[e] = v;
            g.a[list[e]] = v;
        }
    }
}

// Realised alignment of every record, ahead of gate_kernel<false>: a warp per record.
__global__ void __launch_bounds__(256) align_kernel(GateArgs g) {
    const int r = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    pdl_wait();
    pdl_launch_dependents();
    if (r >= g.R) return;
    if (g.keep && !g.keep[r]) {
        if (lane == 0) g.a[r] = __int_as_float(0x7fc00000);
        return;
    }
    const float sv = lane < g.rank ? g.s[(size_t)r * g.rank + lane] : 0.f;
    const float xv = lane < g.rank ? g.xi[(size_t)r * g.rank + lane] : 0.f;
    const float dot = warp_sum(sv * xv), ns = sqrtf(warp_sum(sv * sv)), nx = sqrtf(warp_sum(xv * xv));
    if (lane == 0) g.a[r] = (ns > 0.f && nx > 0.f) ? dot / (ns * nx) : 0.f;
}

// A CTA per slot: its records, in order, go into the running moments; then the score and the gate, with the RMS of the
// memory row.  Bound by latency: all threads look for the slot's records (512 at a time) and have the memory row's loads
// in flight meanwhile (a warp per slot took 14 us for 512 slots and records of d 3584).
// FEW (at most GATE_FEW records, all looked at in one go): a record's alignment is formed by the warp that finds it, and those of
// no slot are shared among the CTAs.  (Formed one at a time, and by the first CTA those of no slot: 512 in one slot 121 us, of none 68.)
template <bool FEW>
__global__ void __launch_bounds__(gt::GATE_THREADS) gate_kernel(GateArgs g, int stray_mask) {
    using namespace gt;
    constexpr int WARPS = GATE_THREADS / 32, MOST = FEW ? GATE_FEW : GATE_BATCH, PER_WARP = MOST / WARPS, GROUPS = MOST / GATE_THREADS;
    __shared__ int hit[MOST];  // FEW: PER_WARP of every warp
    __shared__ float val[MOST];
    __shared__ int n_hit, n_own[WARPS];
    __shared__ float red[WARPS];
    const int j = blockIdx.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    pdl_wait();
    pdl_launch_dependents();
    if (tid == 0) n_hit = 0;
    int sl[GROUPS];
    // FEW: a warp has consecutive records, the same number of groups of 32 each
    const int groups = (g.R + GATE_THREADS - 1) / GATE_THREADS, rw = warp * groups * 32 + lane;
    if (FEW)
#pragma unroll
        for (int q = 0; q < GROUPS; ++q) sl[q] = q < groups && rw + 32 * q < g.R ? g.slot[rw + 32 * q] : 0;
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
    auto moment = [&](float v) {
        n += 1;
        const float delta = v - mean;
        mean += delta / (float)n;
        M2 += delta * (v - mean);
        nfb += 1;
    };
    if (FEW) {
        int *const list = hit + warp * PER_WARP;  // this slot's records in order; from the end, those of no slot
        int own_n = 0, none_n = 0;
#pragma unroll
        for (int q = 0; q < GROUPS; ++q) {
            const int r = rw + 32 * q;
            // (a record of no slot of this call has an alignment all the same)
            bool own = sl[q] == j, none = (unsigned)sl[q] >= (unsigned)g.S && (r & stray_mask) == j;
            if (q >= groups || !__any_sync(0xffffffffu, r < g.R && (own || none))) continue;
            own = own && r < g.R;
            none = none && r < g.R;
            if ((own || none) && g.keep && !g.keep[r]) {
                g.a[r] = __int_as_float(0x7fc00000);
                own = none = false;
            }
            const unsigned mo = __ballot_sync(0xffffffffu, own), mn = __ballot_sync(0xffffffffu, none), below = (1u << lane) - 1u;
            if (own) list[own_n + __popc(mo & below)] = r;
            if (none) list[PER_WARP - 1 - none_n - __popc(mn & below)] = r;
            own_n += __popc(mo);
            none_n += __popc(mn);
        }
        __syncwarp();
        if (own_n == 1) {  // (the usual case, and the shorter code: 512 records in 512 slots 7.0 us in a graph, with the general one 7.8)
            alignments<0>(g, list, 1, val + warp * PER_WARP, lane);
        } else if (own_n > 1) {
            alignments<GATE_RECS_LOG>(g, list, own_n, val + warp * PER_WARP, lane);
        }
        if (none_n > 0) alignments<GATE_RECS_LOG>(g, list + PER_WARP - none_n, none_n, nullptr, lane);
        if (lane == 0) n_own[warp] = own_n;
        __syncthreads();
        if (tid == 0)
            for (int w = 0; w < WARPS; ++w)
                for (int e = 0, ne = n_own[w]; e < ne; ++e) moment(val[w * PER_WARP + e]);
    } else {
        __syncthreads();
        for (int r0 = 0; r0 < g.R; r0 += GATE_BATCH) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int r = r0 + q * GATE_THREADS + tid;
                sl[q] = r < g.R ? g.slot[r] : -1;
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int r = r0 + q * GATE_THREADS + tid;
                if (sl[q] == j && r < g.R && (!g.keep || g.keep[r])) hit[atomicAdd(&n_hit, 1)] = r;
            }
            __syncthreads();
            const int nh = n_hit;
            __syncthreads();  // (all have read it before the next records are counted)
            if (nh == 0) continue;
            // in record order
            for (int e = tid; e < nh; e += GATE_THREADS) {
                const int r = hit[e];
                int rk = 0;
                for (int f = 0; f < nh; ++f) rk += hit[f] < r;
                val[rk] = g.a[r];
            }
            __syncthreads();
            if (tid == 0) {
                n_hit = 0;
                for (int e = 0; e < nh; ++e) moment(val[e]);
            }
            __syncthreads();
        }
    }
    ss = warp_sum(ss);
    if (lane == 0) red[warp] = ss;
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

// Records per cluster, records per warp, columns of four at a time and shared memory of a sketch.
// us, rank 24, records per cluster x per warp:          8 x 1   8 x 2   8 x 4   16 x 2   16 x 4
//   d 256:   64 / 296 / 1024 / 4096 records    4.4   4.1   4.6   4.9   4.7 | 4.9 4.7 5.5 4.9 4.8 | 6.5 6.8 10.7 5.9 7.1 | 22.9 21.1 29.9 14.4 17.8
//   d 1536:  64 / 296 / 1024 / 2048            5.6   4.7   5.0   6.2   6.0 | 6.9 5.8 6.3 6.3 6.0 | 10.5 9.0 12.1 9.7 9.7 | 19.6 16.3 19.9 18.1 15.1
//   d 3584:  64 / 264 / 272 / 512              7.6   6.2   6.2   8.9   8.1 | 9.3 6.5 6.6 9.1 8.2 | 10.8 11.4 11.6 9.0 8.2 | 11.3 12.1 12.2 9.2 8.4
// Few records: eight per cluster, for more CTAs.  33 clusters fit side by side at a CTA per SM, and 37 where two fit an SM.
// More: sixteen halve the reads of Pi.  Four per warp take more registers (three CTAs per SM), so where shared memory leaves room for
// more CTAs than that, two per warp.
struct SketchForm {
    int per, vpw, cols, bytes;
};
static SketchForm sketch_form(int R, int d, int rank) {
    using namespace gt;
    const int cols_all = (d / 4 + SK_CLUSTER - 1) / SK_CLUSTER;
    auto with = [&](int per, int vpw) {
        const int cols = std::min(cols_all, SK_SMEM / 16 / (rank + per));
        return SketchForm{per, vpw, cols, (rank + per) * cols * 16};
    };
    // CTAs that an SM holds: shared memory with the partial products and what the system keeps, `most` by registers
    auto fit = [](const SketchForm &f, int most) {
        const int parts = SK_WARPS / (f.per / f.vpw) * f.per * MAX_RANK * 4;
        return std::min(most, 228 * 1024 / (f.bytes + parts + 1024));
    };
    const SketchForm few = with(8, 2), two = with(16, 2), four = with(16, 4);
    if (R <= (fit(few, 4) >= 2 ? 8 * 37 : 8 * 33)) return few;
    return fit(four, 3) == fit(two, 4) ? four : two;
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
        const SketchForm f = sketch_form(R, d, rank);
        auto *const kern = f.per == 8 ? sketch_kernel<8, 2> : f.vpw == 2 ? sketch_kernel<16, 2> : sketch_kernel<16, 4>;
        const int rc = device_setup(reinterpret_cast<const void *>(kern), gt::SK_SMEM, nullptr);
        if (rc != SPECROLL_OK) return rc;
        SR_CUDA_TRY(launch_clusters(true, gt::SK_CLUSTER, kern, dim3((unsigned)((R + f.per - 1) / f.per * gt::SK_CLUSTER)),
                                    dim3(gt::SK_THREADS), (size_t)f.bytes, st, R, d / 4, rank, f.cols,
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
    // more than GATE_FEW records: the alignments are needed by the second kernel, and the caller's array is where they are kept
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
    if (d->R > gt::GATE_FEW) {
        SR_CUDA_TRY(launch_dependent(true, align_kernel, dim3((unsigned)(d->R + 7) / 8), dim3(256), 0, st, g));
        SR_CUDA_TRY(launch_dependent(true, gate_kernel<false>, dim3((unsigned)d->S), dim3(gt::GATE_THREADS), 0, st, g, 0));
        return SPECROLL_OK;
    }
    int share = 1;  // CTAs that share the records of no slot: a power of two
    while (share <= d->S / 2) share *= 2;
    SR_CUDA_TRY(launch_dependent(true, gate_kernel<true>, dim3((unsigned)d->S), dim3(gt::GATE_THREADS), 0, st, g, share - 1));
    return SPECROLL_OK;
}
