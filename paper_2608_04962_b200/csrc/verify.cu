// Exact target verification: softmax statistics of every tree node, the node-wise
// accept / resample walk, and the terminal (fallback or bonus) draw.
//
// Two launches per plain call:
//   row_stats_kernel    (few rows: run_stats_kernel) streams the bf16 logits once, an online (max, sum-exp)
//                       pair per thread, and leaves the pair of every eighth of every (sequence, node) row.
//   walk_term_kernel    one CTA (or cluster) per sequence, launched to overlap the tail of the
//                       statistics kernel: the walk, then the terminal draw.  The residual of the
//                       walk differs from p only on the <= k candidates of the current node (the
//                       proposal is zero elsewhere), so it is tracked as k numbers plus one scale
//                       for the rest of the vocabulary, all in fp64; the terminal draw is an
//                       inverse CDF over the vocabulary in token order with fp64 segment sums, the
//                       walk's <= k residual entries overriding the plain softmax mass.
// Logits that were never stored: the same kernel with the projection's numbers (wanted logits, tile masses) in
// place of the rows.  Statistics only of visited rows, and nucleus targets: walk_cta_kernel, walk and draw too.  The steps
// one by one, for logits that were never stored: walk_kernel and terminal_kernel.
#include <math.h>

#include <algorithm>
#include <mutex>

#include "common.cuh"
#include "tc05.cuh"

namespace specroll {

SR_CHECK_TU()

constexpr int RS_THREADS = 256;
constexpr int WALK_WARPS = 4;
constexpr int TERM_THREADS = 512;  // two CTAs per SM
constexpr int TERM_WARPS = TERM_THREADS / 32;
constexpr int TERM_SMEM_LIMIT = 200 * 1024;  // slice masses of the terminal draw by one CTA
constexpr int WALK_CTA_SMEM = 220 * 1024;    // the same and the staged walk
constexpr float NEG_INF = -INFINITY;

// ------------------------------------------------------------------------------ row statistics

// nmc = -m c rides along with the running maximum m, so that an exponent is one fused multiply-add.
__device__ __forceinline__ void online_update(const uint4 &v, float c, float &m, float &nmc, float &s) {
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
    float x[8];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        x[2 * i] = __uint_as_float(w[i] << 16);
        x[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
    }
    float vm = x[0];
#pragma unroll
    for (int i = 1; i < 8; ++i) vm = fmaxf(vm, x[i]);
    if (vm > m) {
        s *= ex2_approx((m - vm) * c);  // m = -inf gives 0
        m = vm;
        nmc = -vm * c;
    }
    float acc = 0.f;
#pragma unroll
    for (int i = 0; i < 8; ++i) acc += ex2_approx(fmaf(x[i], c, nmc));
    s += acc;
}

// Four vectors in turn with the same result to the last bit, for a warp that has its scheduler to itself: the four sums of
// exponentials are independent of one another once the maxima are known, and nothing branches.
__device__ __forceinline__ void online_update4(const uint4 (&v)[4], float c, float &m, float &nmc, float &s) {
    float f[4], acc[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const uint32_t w[4] = {v[q].x, v[q].y, v[q].z, v[q].w};
        float x[8];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            x[2 * i] = __uint_as_float(w[i] << 16);
            x[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
        }
        const float vm = fmaxf(fmaxf(fmaxf(x[0], x[1]), fmaxf(x[2], x[3])), fmaxf(fmaxf(x[4], x[5]), fmaxf(x[6], x[7])));
        const bool up = vm > m;
        f[q] = up ? ex2_approx((m - vm) * c) : 1.f;
        nmc = up ? -vm * c : nmc;
        m = up ? vm : m;
        acc[q] = 0.f;
#pragma unroll
        for (int i = 0; i < 8; ++i) acc[q] += ex2_approx(fmaf(x[i], c, nmc));
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) s = __fadd_rn(__fmul_rn(s, f[q]), acc[q]);
}

// logits[rows, V] bf16; c = log2(e) / T.  row_max = max_v l_v, row_sum = sum_v exp((l_v - max)/T).
// The row is cut into groups of 128 8-token vectors; a warp takes one contiguous run of groups and reads a group
// with four loads of 32 consecutive vectors (2 KB in one piece per warp).  32 registers, so that eight CTAs fit an SM.
constexpr int RS_WARPS = RS_THREADS / 32;

// The run of 8-token vectors that warp w of the statistics kernel takes of a row of nvec vectors, [v_lo, v_hi).
__host__ __device__ inline void rs_run(int nvec, int w, int *v_lo, int *v_hi) {
    const int G = (nvec + 127) / 128, gpw = (G + RS_WARPS - 1) / RS_WARPS;
    const int g_lo = w * gpw < G ? w * gpw : G, g_hi = g_lo + gpw < G ? g_lo + gpw : G;
    *v_lo = g_lo * 128 < nvec ? g_lo * 128 : nvec;
    *v_hi = g_hi * 128 < nvec ? g_hi * 128 : nvec;
}
__host__ __device__ inline int rs_run_of_vec(int nvec, int vi) {
    const int G = (nvec + 127) / 128, gpw = (G + RS_WARPS - 1) / RS_WARPS;
    return (vi / 128) / gpw;
}

// Maximum and sum of a run [v_lo, v_hi) by one warp, in groups of 128 vectors.
__device__ __forceinline__ void run_stats(const uint4 *__restrict__ p, int nvec, int v_lo, int v_hi, int lane, float c, float &m, float &s) {
    float nmc = 0.f;
    m = NEG_INF;
    s = 0.f;
#pragma unroll 1
    for (int i0 = v_lo + lane; i0 - lane < v_hi; i0 += 128) {
        if (i0 + 3 * 32 < nvec) {  // (for lane 31: the whole group is inside the row)
            uint4 v[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) v[q] = ld_nc_v4(p + i0 + q * 32);
#pragma unroll
            for (int q = 0; q < 4; ++q) online_update(v[q], c, m, nmc, s);
        } else {
            for (int q = 0; q < 4; ++q)
                if (i0 + q * 32 < nvec) online_update(ld_nc_v4(p + i0 + q * 32), c, m, nmc, s);
        }
    }
    const float mw = warp_max(m);
    s = (m == NEG_INF) ? 0.f : s * ex2_approx((m - mw) * c);
    s = warp_sum(s);
    m = mw;
}

// A row's own pair from its runs' pairs, by warp 0 of a CTA.
__device__ __forceinline__ void row_from_runs(const float2 *sh, int lane, float c, float *row_max, float *row_sum) {
    const float2 e = lane < RS_WARPS ? sh[lane] : make_float2(NEG_INF, 0.f);
    const float mb = warp_max(e.x);
    const float s = warp_sum(e.x == NEG_INF ? 0.f : e.y * ex2_approx((e.x - mb) * c));
    if (lane == 0) {
        *row_max = mb;
        *row_sum = s;
    }
}

// run_tab: [rows][RS_WARPS] (m, s) of every run of every row, s = sum over the run of exp((l - m)/T).  The kernel that
// walks adds a row's pairs up; the terminal draw finds the eighth of the row that holds its target from them and reads
// only that.  This is the form for few rows: a warp takes a run, or a few in turn, through a ring of bulk copies of 2 KB
// (with its loads in registers a warp has 2 KB in flight, so a run is 19 dependent rounds however empty the machine); the
// ring is as deep as the CTAs of an SM leave room for.  The terms of a lane's sum keep the order that the CTA-per-row form
// (row_stats_kernel) gives them: the terminal draw follows the last bits of the runs' sums.
constexpr int RUN_PIECE = 128;                 // vectors per copy (a group)
constexpr int RUN_RING_MIN = 2, RUN_RING_MAX = 10;  // copies in flight per warp
constexpr int RUN_WARPS = 4;                   // warps per CTA
constexpr int RUN_CTAS = 8, RUN_CTAS_MORE = 11;  // CTAs per SM: the fewer, with deeper rings, or as many as give every run a warp
// ROWS: a CTA of eight warps takes the eight runs of row blockIdx and leaves the row's own pair (up to four rows per SM).
#ifdef SPECROLL_CHECK
// Debug build only: when armed (specroll_check_inject(2)), the first warp of CTA 0 leaves out its first copy, once.  Its wait runs
// into the time limit; the copies behind it land before the CTA goes away.
static __device__ int g_drop_one_copy;
int run_stats_arm_dropped_copy() {
    const int one = 1;
    return cudaMemcpyToSymbol(g_drop_one_copy, &one, sizeof(one)) == cudaSuccess ? SPECROLL_OK : SPECROLL_ECUDA;
}
#else
int run_stats_arm_dropped_copy() { return -1; }
#endif
template <bool ROWS, int CTAS>
__global__ void __launch_bounds__(32 * (ROWS ? RS_WARPS : RUN_WARPS), CTAS)
run_stats_kernel(const uint16_t *__restrict__ logits, int V, float c, int n_runs, int ring_n, float2 *__restrict__ run_tab,
                 float *__restrict__ row_max, float *__restrict__ row_sum) {
    constexpr int WARPS = ROWS ? RS_WARPS : RUN_WARPS;
    extern __shared__ __align__(128) uint4 ring_all[];  // [WARPS][ring_n][RUN_PIECE]
    __shared__ __align__(8) unsigned long long full_all[WARPS][RUN_RING_MAX];
    __shared__ volatile int abort_all[WARPS];
    __shared__ float2 sh[RS_WARPS];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nvec = V >> 3;
    const int first = ROWS ? blockIdx.x * RS_WARPS + warp : warp * gridDim.x + blockIdx.x, stride = ROWS ? n_runs : RUN_WARPS * gridDim.x;
    uint4 *ring = ring_all + (size_t)warp * ring_n * RUN_PIECE;
    unsigned long long *full = full_all[warp];
    volatile int *abort_flag = &abort_all[warp];
    if (lane == 0) {
        for (int s = 0; s < ring_n; ++s) mbar_init(smem_u32(&full[s]), 1);
        *abort_flag = 0;
        fence_mbar_init();
    }
    __syncwarp();
    // Set up under the tail of the kernel before, which may have written the logits.  The kernel launched behind this
    // one as its programmatic dependent reads the call's other inputs before it waits for the statistics: it may only
    // start once everything in front of this kernel is complete.
    pdl_wait();
    pdl_launch_dependents();
    // the copies ahead: run, and vector within it
    int r_next = first, v_next = 0, v_end = 0;
    uint32_t n_issued = 0, n_used = 0;
    int s_in = 0, s_out = 0;    // slots of the next copy and of the next piece to use
    uint32_t phase = 0;         // parity of s_out's round
    auto bounds = [&](int r, int *lo, int *hi) { rs_run(nvec, r % RS_WARPS, lo, hi); };
    auto skip_empty = [&]() {  // (a run of a short row may be empty)
        while (r_next < n_runs) {
            bounds(r_next, &v_next, &v_end);
            if (v_next < v_end) return;
            r_next += stride;
        }
    };
    auto issue = [&]() {
        if (r_next >= n_runs) return;
        const int n = min(RUN_PIECE, v_end - v_next);
        if (lane == 0) {
            const uint32_t bar = smem_u32(&full[s_in]);
            mbar_arrive_expect_tx(bar, (uint32_t)n * 16u);
            bool copy = true;
#ifdef SPECROLL_CHECK
            if (blockIdx.x == 0 && warp == 0 && n_issued == 0 && atomicExch(&g_drop_one_copy, 0) == 1) copy = false;
#endif
            if (copy) bulk_load(smem_u32(ring + s_in * RUN_PIECE), reinterpret_cast<const uint4 *>(logits + (size_t)(r_next / RS_WARPS) * V) + v_next,
                      (uint32_t)n * 16u, bar);
        }
        ++n_issued;
        if (++s_in == ring_n) s_in = 0;
        v_next += n;
        if (v_next >= v_end) {
            r_next += stride;
            skip_empty();
        }
    };
    skip_empty();
    for (int s = 0; s < ring_n; ++s) issue();
    bool ok = true;
    for (int r = first; r < n_runs; r += stride) {
        int v_lo, v_hi;
        bounds(r, &v_lo, &v_hi);
        float m = NEG_INF, nmc = 0.f, s = 0.f;
        for (int v0 = v_lo; v0 < v_hi && ok; v0 += RUN_PIECE) {
            ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&full[s_out]), phase, abort_flag));
            if (!ok) break;
            const uint4 *p = ring + s_out * RUN_PIECE + lane;
            const int n = v_hi - v0 - lane;
#pragma unroll
            for (int g = 0; g < RUN_PIECE / 128; ++g) {
                uint4 v[4];
                if (g * 128 + 128 <= v_hi - v0) {
#pragma unroll
                    for (int q = 0; q < 4; ++q) v[q] = p[g * 128 + q * 32];
                    online_update4(v, c, m, nmc, s);
                } else {
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        if (g * 128 + q * 32 < n) online_update(p[g * 128 + q * 32], c, m, nmc, s);
                }
            }
            ++n_used;
            if (++s_out == ring_n) {
                s_out = 0;
                phase ^= 1u;
            }
            __syncwarp();
            if (lane == 0) fence_proxy_async();  // the piece has been read before the copy engine writes its place again
            issue();
        }
        const float mw = warp_max(m);
        s = (m == NEG_INF) ? 0.f : s * ex2_approx((m - mw) * c);
        s = warp_sum(s);
        // (a copy that does not arrive: cannot happen with readable logits; this run and those after it are marked instead of
        // left looking valid)
        const float2 e = ok ? make_float2(mw, s) : make_float2(nanf(""), nanf(""));
        if (lane == 0) {
            if (ROWS)
                sh[warp] = e;
            else
                run_tab[r] = e;
        }
    }
    if (!ok && lane == 0) {  // let the copies still in flight land before the CTA goes away
        for (uint32_t i = n_used; i < n_issued; ++i) {
            const unsigned long long t0 = globaltimer_ns();
            while (!mbar_try_wait(smem_u32(&full[i % ring_n]), (i / ring_n) & 1u) && globaltimer_ns() - t0 < 100000000ull) {
            }
        }
    }
    if (ROWS) {
        __syncthreads();
        if (warp == 0) row_from_runs(sh, lane, c, row_max + blockIdx.x, row_sum + blockIdx.x);
    }
}

// A CTA per row: the pairs of the row's runs to run_tab, or (run_tab null) the row's own pair.
__global__ void __launch_bounds__(RS_THREADS, 8)
row_stats_kernel(const uint16_t *__restrict__ logits, int V, float c, float *__restrict__ row_max, float *__restrict__ row_sum,
                 float2 *__restrict__ run_tab) {
    pdl_wait();  // (as in run_stats_kernel)
    pdl_launch_dependents();
    __shared__ float2 sh[RS_WARPS];
    const size_t row = blockIdx.x;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nvec = V >> 3;
    int v_lo, v_hi;
    rs_run(nvec, warp, &v_lo, &v_hi);
    float m, s;
    run_stats(reinterpret_cast<const uint4 *>(logits + row * (size_t)V), nvec, v_lo, v_hi, lane, c, m, s);
    if (run_tab) {
        if (lane == 0) run_tab[row * RS_WARPS + warp] = make_float2(m, s);
        return;
    }
    if (lane == 0) sh[warp] = make_float2(m, s);
    __syncthreads();
    if (warp == 0) row_from_runs(sh, lane, c, row_max + row, row_sum + row);
}

// ------------------------------------------------------------------------------ nucleus threshold

// Order-preserving 16-bit key of a bf16 value (-0 counts as +0): larger value <=> larger key.
__device__ __forceinline__ uint32_t ord_key(uint32_t bits) {
    if (bits == 0x8000u) bits = 0u;
    return (bits & 0x8000u) ? (~bits & 0xffffu) : (bits | 0x8000u);
}

constexpr int NUC_THREADS = 512;

// Nucleus of one row (sampling configuration of the experiments: threshold 0.95): tokens are taken in order of
// decreasing probability until their mass first reaches top_p, and every token that ties with the last one
// taken is kept too.  Equal probabilities are equal bf16 logits, so the kept set is "key >= threshold key".
// Run by all NUC_THREADS threads of a CTA; the row comes from HBM or L2 once.  Result: st->prefix = threshold key (a
// token is kept iff ord_key(logit) >= key), st->keep = sum of the kept exp((l - M)/T).
//
// A token's mass depends on its 16 bits alone, so one pass COUNTS the tokens of every bf16 value in shared memory and
// the cut is found from the counts alone, values in falling order (nucleus_cut).  Only tokens at or above a bound are
// counted: all tokens below M - T ln(V / ((1 - top_p) S)) together weigh at most (1 - top_p) S, so the cut lies at or above it,
// and peaked rows count a few tokens.  What the pass waits for is the count: a warp's shared-memory atomic takes five to six
// cycles of the SM whether twelve or twenty-four of its lanes count (with the integer instructions of the addresses about
// 15 k cycles for a row of 152 k tokens; loads a round ahead do not help, nor does a closer bound from a sample).  Where a
// counter does not tell the values apart, or the counted mass stays below the target by rounding, the radix search over the
// whole row gives the same result in four passes (nucleus_row_radix).  Verification of 256 sequences x 16 nodes, V 151936:
// 590 us with a search of two passes over the tokens per row, 349 us with this one.
constexpr int NUC_OCT_LO = (127 - 13) << 7;              // bf16 bits of 2^-13
constexpr int NUC_VALUES = ((127 + 15) << 7) - NUC_OCT_LO;  // counters per sign; 0: nearer to zero than 2^-13
constexpr int NUC_SIGN = 8192;                           // the negative values' table, 2^15 bytes behind the other: the sign bit of a
                                                         // 16-bit word is an address bit
constexpr int NUC_BASE_MAX = 0x8000 - 4 * NUC_VALUES;    // largest address of the tables for which that is so

struct NucleusSmem {
    union {
        uint32_t count[NUC_SIGN + NUC_VALUES];
        float bins[16][NUC_THREADS];
    };
    float wsum[NUC_THREADS / 32][16];
    unsigned long long wtot[NUC_THREADS / 32];
    unsigned long long upto, inside;  // fixed-point mass up to and including the place of the cut; of its bin down to there
    int last;      // place at which the fixed-point mass from the top reaches the target, -1: nowhere
    uint32_t k_min, k_max;            // the bin's keys
    int p_min, p_max;                 // its places
    float digit[16];
    int sel;       // bin selected by the last level
    float above, keep;
    uint32_t prefix;
};

// Sums the sixteen private bins over the block; thread 0 then picks, from the first bin on, the bin at which
// above + running mass reaches the target (or the last bin with mass if rounding keeps the total below it) and
// leaves it in st->sel, the mass before it in st->above and the mass up to and including it in st->keep.
__device__ void nucleus_pick(NucleusSmem *st, float target, bool top_is_high_index) {
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
#pragma unroll
    for (int j = 0; j < 16; ++j) {
        const float x = warp_sum(st->bins[j][tid]);
        if (lane == 0) st->wsum[warp][j] = x;
    }
    __syncthreads();
    if (warp == 0) {
        // lane j adds bin j over the warps (in warp order); lane 0 then walks the sixteen totals
        float x = 0.f;
        if (lane < 16)
            for (int w2 = 0; w2 < NUC_THREADS / 32; ++w2) x += st->wsum[w2][lane];
        float tot[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) tot[j] = __shfl_sync(0xffffffffu, x, top_is_high_index ? 15 - j : j);  // tot[0] = most probable bin
        if (lane == 0) {
            float cum = st->above;
            int sel = -1, last = 0;
#pragma unroll
            for (int j = 0; j < 16; ++j)
                if (tot[j] > 0.f) last = j;
#pragma unroll
            for (int j = 0; j < 16; ++j) {
                if (sel < 0) {
                    if (cum + tot[j] >= target)
                        sel = j;
                    else
                        cum += tot[j];
                }
            }
            float tsel = 0.f;
            if (sel < 0) {
                sel = last;
                cum = st->above;
#pragma unroll
                for (int j = 0; j < 16; ++j)
                    if (j < last) cum += tot[j];
            }
#pragma unroll
            for (int j = 0; j < 16; ++j)
                if (j == sel) tsel = tot[j];
            st->above = cum;
            st->keep = cum + tsel;
            st->sel = top_is_high_index ? 15 - sel : sel;
        }
    }
    __syncthreads();
}

// One radix pass of the key search: masses of the keys whose leading bits equal `prefix`, by their next four bits.
__device__ __forceinline__ void nucleus_key_bin(NucleusSmem *st, uint32_t bits, int level, uint32_t prefix, float M,
                                                float c) {
    const int shift = 12 - 4 * level;
    const uint32_t key = ord_key(bits);
    if (level == 0 || (key >> (shift + 4)) == prefix)
        st->bins[(key >> shift) & 15u][threadIdx.x] += ex2_approx((__uint_as_float(bits << 16) - M) * c);
}

// Exact search over the whole row (fallback): four passes, four key bits each.
__device__ void nucleus_row_radix(const uint4 *__restrict__ p, int nvec, float c, float M, float target,
                                  NucleusSmem *st) {
    const int tid = threadIdx.x;
    if (tid == 0) {
        st->above = 0.f;
        st->prefix = 0u;
    }
    __syncthreads();
    for (int level = 0; level < 4; ++level) {
        const uint32_t prefix = st->prefix;
#pragma unroll
        for (int j = 0; j < 16; ++j) st->bins[j][tid] = 0.f;
        for (int i = tid; i < nvec; i += NUC_THREADS) {
            const uint4 v = ld_nc_v4(p + i);
            const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int t = 0; t < 8; ++t)
                nucleus_key_bin(st, (t & 1) ? (w[t >> 1] >> 16) : (w[t >> 1] & 0xffffu), level, prefix, M, c);
        }
        nucleus_pick(st, target, true);
        if (tid == 0) st->prefix = (prefix << 4) | (uint32_t)st->sel;
        __syncthreads();
    }
}

// One counter more for the tokens of a pair of bf16 logits that are at or above the bound (lo2: the bound, twice).
// base: the shared-memory address of the tables (in a cluster its upper half holds the CTA's rank), base2: its lower half,
// twice.  The pass is bound by the integer pipe and the atomics: six integer instructions per pair.
__device__ __forceinline__ void nucleus_count2(uint32_t w, uint32_t lo2, uint32_t base, uint32_t base2) {
    // the magnitude's steps above 2^-13, within the table (a counted token lies below 2^15)
    const uint32_t mag = __viaddmin_s16x2_relu(w & 0x7fff7fffu, (uint32_t)(-NUC_OCT_LO & 0xffff) * 0x10001u, (NUC_VALUES - 1) * 0x10001u);
    const uint32_t at = (mag * 4u + base2) | (w & 0x80008000u);
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ge.bf16x2 p|q, %0, %1;\n\t"
        "@p red.shared.add.u32 [%2], 1;\n\t"
        "@q red.shared.add.u32 [%3], 1;\n\t}" ::"r"(w),
        "r"(lo2), "r"(__byte_perm(at, base, 0x7610)), "r"(__byte_perm(at, base, 0x7632))
        : "memory");
}

// A place is a counter's rank by falling value, 0 = the largest positive one, NUC_ZERO = the counter around zero.
constexpr int NUC_ZERO = NUC_VALUES - 1;
__device__ __forceinline__ int nucleus_place(uint32_t bits) {
    const int m = max((int)(bits & 0x7fffu) - NUC_OCT_LO, 0);
    return (bits & 0x8000u) ? NUC_ZERO + m : NUC_ZERO - m;
}
__device__ __forceinline__ uint32_t nucleus_value(int r) {  // (bf16 bits; the counter around zero: 0)
    return r < NUC_ZERO ? (uint32_t)(NUC_ZERO - r + NUC_OCT_LO) : r > NUC_ZERO ? (uint32_t)(r - NUC_ZERO + NUC_OCT_LO) | 0x8000u : 0u;
}
__device__ __forceinline__ uint32_t nucleus_count_at(const NucleusSmem *st, int r) {
    const int at = r <= NUC_ZERO ? NUC_ZERO - r : NUC_SIGN + r - NUC_ZERO;
    return st->count[at] + (r == NUC_ZERO ? st->count[NUC_SIGN] : 0u);
}

// The cut, from the counts of the places [r0, r1], by all threads of a CTA; false: it is not resolved by the counts.
//   1  The place at which the mass from the top reaches the target, masses as 32-bit fixed point (the row's largest element is
//      2^32), exact integer sums.  It names a bin of the distance below the maximum, 1/8 unit of log2 wide.
//   2  Within the bin the cut is found digit by digit over the 16-bit key, in fp32 from the mass above the bin on.
// (The steps of a search that adds up the tokens themselves, first in bins and then by digits: the cut follows the rounding
// of its sums where a cumulative mass lies within 1e-7 of the target, so the arithmetic is the same.)
__device__ bool nucleus_cut(NucleusSmem *st, int r0, int r1, float M, float c, float target) {
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const float Mc = M * c;
    auto dist = [&](uint32_t bits) { return Mc - __uint_as_float(bits << 16) * c; };
    auto bin = [&](float e) { return (int)(__float_as_uint(e * 8.0f + 12582912.0f) - 0x4B400000u); };  // (rounded to nearest)
    auto fixed_at = [&](int r) {
        const uint32_t n = nucleus_count_at(st, r);
        if (n == 0u) return 0ull;
        const float e = dist(nucleus_value(r));
        return bin(e) < 256 ? (unsigned long long)n * __float2uint_rn(ex2_approx(-e) * 4294967296.0f) : 0ull;
    };
    // A warp has consecutive places, a lane every 32nd of them: beside another CTA that counts, accesses to shared memory are what
    // this waits for.  (A thread's places next to one another, eight lanes to a bank, and one thread going through the
    // digits took 8 us a row: verification of 8 / 64 / 256 sequences 73 / 163 / 358 us, now 70 / 160 / 349.)
    auto sum_u64 = [&](unsigned long long v) {  // over a warp (a sum below 2^59)
        return ((unsigned long long)__reduce_add_sync(0xffffffffu, (uint32_t)(v >> 27)) << 27) +
               __reduce_add_sync(0xffffffffu, (uint32_t)v & 0x7ffffffu);
    };
    const unsigned long long tgt = (unsigned long long)((double)target * 4294967296.0);
    const int per = (r1 - r0 + NUC_THREADS) / NUC_THREADS;  // (<= 14)
    const int w0 = r0 + warp * 32 * per, w1 = min(r1 + 1, w0 + 32 * per);
    unsigned long long part = 0ull;
    for (int r = w0 + lane; r < w1; r += 32) part += fixed_at(r);
    part = sum_u64(part);
    if (lane == 0) st->wtot[warp] = part;
    if (tid == 0) {
        st->last = -1;
        st->inside = 0ull;
        st->k_min = 0xffffu;
        st->k_max = 0u;
        st->p_min = 0x7fffffff;
        st->p_max = -1;
    }
    __syncthreads();
    unsigned long long cum64 = sum_u64(lane < warp ? st->wtot[lane] : 0ull);
    if (cum64 < tgt && cum64 + part >= tgt) {  // (one warp at most)
        for (int r = w0 + lane;; r += 32) {
            unsigned long long v = r < w1 ? fixed_at(r) : 0ull;
            const unsigned long long all = sum_u64(v);
            if (cum64 + all < tgt) {
                cum64 += all;
                continue;
            }
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned long long x = __shfl_up_sync(0xffffffffu, v, o);
                if (lane >= o) v += x;
            }
            const unsigned hit = __ballot_sync(0xffffffffu, cum64 + v >= tgt);
            if (lane == __ffs(hit) - 1) {
                st->last = r;
                st->upto = cum64 + v;
            }
            break;
        }
    }
    __syncthreads();
    const int last = st->last;
    if (last < 0) return false;
    const int jb = bin(dist(nucleus_value(last)));
    // the places of the bin (the bins do not fall from place to place)
    const bool here = w0 < w1 && bin(dist(nucleus_value(w0))) <= jb && bin(dist(nucleus_value(w1 - 1))) >= jb;
    if (here) {
        unsigned long long in = 0ull;
        uint32_t lo = 0xffffu, hi = 0u;
        int b_min = 0x7fffffff, b_max = -1;
        for (int r = w0 + lane; r < w1; r += 32) {
            if (bin(dist(nucleus_value(r))) != jb) continue;
            b_min = min(b_min, r);
            b_max = r;
            if (nucleus_count_at(st, r) == 0u) continue;
            if (r <= last) in += fixed_at(r);
            const uint32_t key = ord_key(nucleus_value(r));
            lo = min(lo, key);
            hi = max(hi, key);
        }
        in = sum_u64(in);
        lo = __reduce_min_sync(0xffffffffu, lo);
        hi = __reduce_max_sync(0xffffffffu, hi);
        b_min = __reduce_min_sync(0xffffffffu, b_min);
        b_max = __reduce_max_sync(0xffffffffu, b_max);
        if (lane == 0) {
            if (in) atomicAdd(&st->inside, in);
            atomicMin(&st->k_min, lo);
            atomicMax(&st->k_max, hi);
            atomicMin(&st->p_min, b_min);
            atomicMax(&st->p_max, b_max);
        }
    }
    __syncthreads();
    const uint32_t k_min = st->k_min, k_max = st->k_max;
    float cum = (float)((double)(st->upto - st->inside) * (1.0 / 4294967296.0));
    float keep = cum;
    uint32_t prefix = 0u;
    // Usually the bin has a few dozen places: their masses side by side in shared memory, and one warp takes the digits' sums, a
    // lane per digit, and goes through them in falling order (with a barrier and an addition in shared memory per digit and
    // thread the digits took 12 k cycles).
    const int p0 = st->p_min, p1 = st->p_max + 1;
    float *const f = &st->wsum[0][0];
    if (p1 - p0 <= (NUC_THREADS / 32) * 16 && (p0 > NUC_ZERO || p1 <= NUC_ZERO)) {  // (all of one sign)
        if (here)
            for (int r = max(p0, w0) + lane; r < min(p1, w1); r += 32)
                f[r - p0] = (float)nucleus_count_at(st, r) * ex2_approx((bf16_bits_to_float(nucleus_value(r)) - M) * c);
        __syncthreads();
        if (warp == 0) {
            const uint32_t key0 = ord_key(nucleus_value(p0));  // (the keys fall by one from place to place)
            int lo = (int)(key0 - k_max), hi = (int)(key0 - k_min) + 1;  // (the places with tokens: at most 17 digits a level)
            for (int shift = 12; shift >= 0; shift -= 4) {
                if (shift > 0 && ((k_min ^ k_max) >> shift) == 0u) continue;
                const int first = (int)((key0 - lo) & ((1u << shift) - 1u)) + 1;  // (places of the first digit, at most)
                const int i = lane == 0 ? lo : min(hi, lo + first + ((lane - 1) << shift));
                const int j = min(hi, lo + first + (lane << shift));
                float sum = 0.f;
#pragma unroll 4
                for (int q = i; q < j; ++q) sum += f[q];
                float t[17];
#pragma unroll
                for (int d = 0; d < 17; ++d) t[d] = __shfl_sync(0xffffffffu, sum, d);
                float run = cum, before = cum, tsel = 0.f;
                int sel = -1;
                bool found = false;
#pragma unroll
                for (int d = 0; d < 17; ++d) {
                    if (found || !(t[d] > 0.f)) continue;
                    sel = d;
                    tsel = t[d];
                    before = run;
                    found = run + t[d] >= target;
                    run += t[d];
                }
                cum = before;  // (none reached the target by rounding: the last digit with mass)
                keep = cum + tsel;
                if (sel >= 0) {
                    hi = __shfl_sync(0xffffffffu, j, sel);
                    lo = __shfl_sync(0xffffffffu, i, sel);
                }
            }
            if (lane == 0) {
                st->prefix = key0 - lo;
                st->keep = keep;
            }
        }
        return true;
    }
    // this thread's places of the bin, [b0, b1)
    const int b0 = max(p0, r0 + tid * per), b1 = min(p1, r0 + (tid + 1) * per);
    for (int level = 0; level < 4; ++level) {
        const int shift = 12 - 4 * level;
        // (one digit for all of the bin: nothing to decide, except the last one's sum)
        if (level < 3 && ((k_min ^ k_max) >> shift) == 0u) {
            prefix = k_min >> shift;
            continue;
        }
        __syncthreads();
        if (tid < 16) st->digit[tid] = 0.f;
        __syncthreads();
        if (__any_sync(0xffffffffu, b1 > b0)) {
            // a thread's places follow one another: a sum per digit, added when the digit changes or, where the warp has one
            // digit, once for the warp
            int dg = -1;
            float sum = 0.f;
            bool several = false;
            for (int r = b0; r < b1; ++r) {
                const uint32_t n = nucleus_count_at(st, r), bits = nucleus_value(r), key = ord_key(bits);
                if (n == 0u || (level > 0 && (key >> (shift + 4)) != prefix)) continue;
                const int d1 = (int)((key >> shift) & 15u);
                if (d1 != dg && dg >= 0) {
                    atomicAdd(&st->digit[dg], sum);
                    sum = 0.f;
                    several = true;
                }
                dg = d1;
                sum += (float)n * ex2_approx((bf16_bits_to_float(bits) - M) * c);
            }
            const int top = __reduce_max_sync(0xffffffffu, dg);
            if (__all_sync(0xffffffffu, !several && (dg == top || dg < 0))) {
                sum = warp_sum(sum);
                if (lane == 0 && top >= 0) atomicAdd(&st->digit[top], sum);
            } else if (dg >= 0) {
                atomicAdd(&st->digit[dg], sum);
            }
        }
        __syncthreads();
        // every thread for itself: digits from the largest on
        float d[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) d[j] = st->digit[15 - j];
        int sel = -1, lastd = 0;
        float run = cum, tsel = 0.f;
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            if (d[j] > 0.f) lastd = j;
            if (sel < 0) {
                if (run + d[j] >= target) {
                    sel = j;
                    tsel = d[j];
                } else {
                    run += d[j];
                }
            }
        }
        if (sel < 0) {  // (rounding kept the total below the target: the last digit with mass)
            sel = lastd;
            run = cum;
#pragma unroll
            for (int j = 0; j < 16; ++j) {
                if (j < lastd) run += d[j];
                if (j == lastd) tsel = d[j];
            }
        }
        cum = run;
        keep = cum + tsel;
        prefix = (prefix << 4) | (uint32_t)(15 - sel);
    }
    if (prefix == 0x8000u) return false;  // (the counter around zero: several values)
    if (tid == 0) {
        st->prefix = prefix;
        st->keep = keep;
    }
    return true;
}

// n_cta > 1: the CTAs of a cluster share the pass, and its first CTA, which alone gets the result, adds their counts;
// the caller has a cluster barrier between two rows.
__device__ void nucleus_row(const uint16_t *__restrict__ row_logits, int V, float c, float M, float S, float top_p,
                            NucleusSmem *st, int n_cta, int rank) {
    const int tid = threadIdx.x;
    const uint4 *p = reinterpret_cast<const uint4 *>(row_logits);
    const int nvec = V >> 3;
    const float target = top_p * S;
    const uint32_t base = smem_u32(st->count);
    // the bound, one bf16 step lower (the rest of its rounding does not matter: a cut that the counted tokens do not reach
    // is searched over the whole row)
    float bound = fmaxf(M - (log2f((float)V) - log2f(S - target)) / c, -32000.0f);
    bound = fminf(bound, M);  // (top_p near 0)
    const uint32_t lo_bits = __bfloat16_as_ushort(__float2bfloat16_rd(bound - 0.008f * fabsf(bound)));
    const bool counted = fabsf(M) < 32000.0f && bf16_bits_to_float(lo_bits) <= M && (base & 0xffffu) <= (uint32_t)NUC_BASE_MAX;
    if (!counted) {  // (uniform over the cluster)
        if (rank == 0) nucleus_row_radix(p, nvec, c, M, target, st);
        return;
    }
    for (int j = tid; j < 2 * NUC_VALUES / 4; j += NUC_THREADS)
        reinterpret_cast<uint4 *>(st->count)[j < NUC_VALUES / 4 ? j : j - NUC_VALUES / 4 + NUC_SIGN / 4] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
    {
        const uint32_t base2 = (base & 0xffffu) * 0x10001u, lob2 = lo_bits * 0x10001u;
        auto count8 = [&](const uint4 &v) {
            nucleus_count2(v.x, lob2, base, base2);
            nucleus_count2(v.y, lob2, base, base2);
            nucleus_count2(v.z, lob2, base, base2);
            nucleus_count2(v.w, lob2, base, base2);
        };
        const int step = NUC_THREADS * n_cta;
        int i = rank * NUC_THREADS + tid;
        for (; i + 3 * step < nvec; i += 4 * step) {
            uint4 v[4];  // four independent loads in flight
#pragma unroll
            for (int q = 0; q < 4; ++q) v[q] = ld_nc_v4(p + i + q * step);
#pragma unroll
            for (int q = 0; q < 4; ++q) count8(v[q]);
        }
        uint4 v[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) v[q] = ld_nc_v4(p + min(i + q * step, nvec - 1));
#pragma unroll
        for (int q = 0; q < 3; ++q)
            if (i + q * step < nvec) count8(v[q]);
    }
    const int r0 = nucleus_place(__float_as_uint(M) >> 16), r1 = nucleus_place(lo_bits);
    if (n_cta > 1) {
        cluster_sync_all();
        // The CTAs' counts into the first CTA's tables, the places spread over the cluster's threads: a counter is read and
        // written by one thread, all its copies in flight together.  (The first CTA adding them up as it scanned, one
        // round trip after the other, took 30 us.)
        auto add_up = [&](uint32_t *at) {
            uint32_t v[8], n = 0;
#pragma unroll
            for (int k = 0; k < 8; ++k) v[k] = k < n_cta ? ld_dsmem_u32(at, k) : 0u;
#pragma unroll
            for (int k = 0; k < 8; ++k) n += v[k];
            st_dsmem_u32(at, 0, n);
        };
        for (int r = r0 + rank * NUC_THREADS + tid; r <= r1; r += n_cta * NUC_THREADS) {
            add_up(st->count + (r <= NUC_ZERO ? NUC_ZERO - r : NUC_SIGN + r - NUC_ZERO));
            if (r == NUC_ZERO) add_up(st->count + NUC_SIGN);
        }
        cluster_sync_all();
        if (rank != 0) return;
    } else {
        __syncthreads();
    }
    bool ok = nucleus_cut(st, r0, r1, M, c, target);  // (the same for all threads)
    // The counter around zero, if it lies above the cut: its values must not differ by more than their mass's rounding.
    if (ok && r0 <= NUC_ZERO && st->last > NUC_ZERO) {
        const double m0 = (double)nucleus_count_at(st, NUC_ZERO) * (double)ex2_approx(-M * c);
        ok = m0 * (double)(c * 0.6931472f) * 0x1p-13 <= 0x1p-25 * (double)S;
    }
    if (!ok) {
        __syncthreads();  // (all have read the counts)
        nucleus_row_radix(p, nvec, c, M, target, st);
    }
    __syncthreads();
}

// ------------------------------------------------------------------------------ walk

struct WalkArgs {
    const uint16_t *logits;
    // sparse form (logits == NULL): the target logits of every node at the candidates of the node's head only,
    // [B, N, k] bf16, as specroll_target_head_stats leaves them
    const uint16_t *cand_target;
    const int32_t *tree_tok;
    const uint8_t *tree_cand;
    const int32_t *cand_id;
    const float *cand_logit;
    const float *u_acc;
    const float *row_max;
    const float *row_sum;
    int32_t *n_acc, *path_node, *out_tok, *term_node, *term_kind;
    float *min_margin;
    // hand-over to the terminal draw
    int32_t *ws_nov;   // [B]    number of override entries (0 for a bonus draw)
    int32_t *ws_ovid;  // [B,k]  token ids whose mass is overridden
    double *ws_ovm;    // [B,k]  their mass, in units where an untouched token v weighs exp((l_v-M)/T)
    int32_t B, N, K, k, V;
    double T;
};

// What a warp carries from node to node of one sequence's walk.
struct WalkState {
    int nacc, kind;
    double sigma;  // residual of a token outside the candidate set = sigma * p(token)
    double p_off;
    float mm;
    bool have_residual;
};

// Per-warp shared scratch of the walk.
struct WalkSmem {
    double r[SPECROLL_MAX_TOPK];
    double w[SPECROLL_MAX_TOPK];
    float cl[SPECROLL_MAX_TOPK];
    int32_t id[SPECROLL_MAX_TOPK];
    double bc[2];  // broadcast slots: current max, accepted flag
    // per child of the node at hand (walk_node): 1 / s_i, the candidates taken before it, its own candidate
    double inv_s[32];
    uint32_t taken[32];
    int32_t jc[32];
};

// Everything the walk of one sequence can read, staged in shared memory in one round of independent loads (the walk on
// its own reads global memory node by node): per node the row's statistics, the acceptance
// uniform, the drawn token and its slot; per head the candidate ids and proposal logits; per walkable node the
// target logits at its head's candidates.
struct WalkStage {
    const float *rmax, *rsum, *uacc;  // [N]
    const int32_t *ttok;              // [N]
    const uint8_t *tcand;             // [N]
    const int32_t *cid;               // [K, k]
    const float *clog;                // [K, k]
    const uint16_t *pre;              // [N, k]
    // optional (nullptr: computed per node): the tree's parent array, the proposal weights exp((c_j - max c)/T) of
    // every head's candidates, the target probabilities of every walkable node's candidates
    const int8_t *parent;  // [N]
    const double *e;       // [K, k]
    const double *p;       // [N, k]
};

__device__ __forceinline__ void walk_begin(const WalkArgs &a, int b, int lane, WalkState *st) {
    st->nacc = 0;
    st->kind = 0;
    st->sigma = 1.0;
    st->p_off = 0.0;
    st->mm = INFINITY;
    st->have_residual = false;
    if (lane == 0) {
        const int K = a.K;
        for (int i = 0; i <= K; ++i) a.path_node[(size_t)b * (K + 1) + i] = a.out_tok[(size_t)b * (K + 1) + i] = -1;
        a.path_node[(size_t)b * (K + 1)] = 0;
    }
}

// One node u (which has children), by one warp: the target's probabilities on the candidates of u's head -
// S is the normaliser and thr the nucleus threshold key (0: none) of u's row - then u's children in slot order.
// Returns the accepted child, or -1 when every child was rejected (the residual is then in sm->r, st->sigma).
// sg (nullable: a.cand_target and the other arrays are read): the sequence's inputs staged in shared memory.
// emit = false: nothing is written to the results and the count of accepted tokens stays (the node is examined
// on its own, before it is known whether the walk reaches it).
__device__ int walk_node_seq(const WalkArgs &a, const Topo &topo, int b, int u, double M, double S, uint32_t thr,
                                           int lane, WalkSmem *sm, WalkState *st, const WalkStage *sg, bool emit) {
    double *r = sm->r, *w = sm->w;
    float *cl = sm->cl;
    int32_t *id = sm->id;
    const int k = a.k, N = a.N, K = a.K;
    const int hd = topo.depth[u];
    const uint16_t *ct = sg ? sg->pre + u * k : a.cand_target + ((size_t)b * N + u) * k;
    // Quotients whose numerator can be exactly zero (the largest logit minus itself, a taken candidate's weight, a
    // residual entry clamped to zero) are formed as products with a reciprocal: a double division with a zero
    // numerator leaves the division's fast path, and one lane on the slow path holds up the whole warp at every slot.
    const double inv_T = 1.0 / a.T, inv_S = 1.0 / S;
    for (int j = lane; j < k; j += 32) {
        const int t = sg ? sg->cid[hd * k + j] : SR_CHECKED(a.cand_id[((size_t)b * K + hd) * k + j], a.V, b);
        id[j] = t;
        cl[j] = sg ? sg->clog[hd * k + j] : a.cand_logit[((size_t)b * K + hd) * k + j];
        const uint32_t bits = ct[j];
        const double l = (double)bf16_bits_to_float((uint16_t)bits);
        r[j] = ord_key(bits) >= thr ? exp((l - M) * inv_T) * inv_S : 0.0;  // r = p_u on the candidates
    }
    __syncwarp();
    // Every lane holds one or two of the k candidates (j = lane, lane + 32); sums and maxima over the candidates
    // are warp reductions, so that the state (sigma, p_off, the margin) is the same in every lane and nothing of
    // the slot loop runs on one lane alone (k-long loops of fp64 divisions on one lane were most of the walk's time).
    st->sigma = 1.0;
    {
        double pc = 0.0;
        for (int j = lane; j < k; j += 32) pc += r[j];
        pc = warp_sum(pc);
        st->p_off = pc < 1.0 ? 1.0 - pc : 0.0;
    }
    uint64_t taken = 0;
    int accepted = -1;
    for (int c = u + 1; c < N && accepted < 0; ++c) {
        if (topo.parent[c] != u) continue;
        // slot proposal q on the candidates not yet taken
        double mx = -INFINITY;
        for (int j = lane; j < k; j += 32)
            if (!((taken >> j) & 1) && (double)cl[j] > mx) mx = (double)cl[j];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        double s = 0.0;
        for (int j = lane; j < k; j += 32) {
            w[j] = ((taken >> j) & 1) ? 0.0 : exp(((double)cl[j] - mx) * inv_T);
            s += w[j];
        }
        s = warp_sum(s);
        const double inv_s = 1.0 / s;
        __syncwarp();
        const int jc = SR_CHECKED((int)(sg ? sg->tcand[c] : a.tree_cand[(size_t)b * N + c]), k, b);
        const double qy = w[jc] * inv_s;
        double ratio;
        if (qy > 0.0)
            ratio = r[jc] > 0.0 ? r[jc] / qy : 0.0;
        else
            ratio = (r[jc] > 0.0) ? INFINITY : 0.0;
        const double uu = (double)(sg ? sg->uacc[c] : a.u_acc[(size_t)b * N + c]);
        const float mg = (float)fabs(uu - ratio);
        if (mg < st->mm) st->mm = mg;
        __syncwarp();
        if (uu < (ratio < 1.0 ? ratio : 1.0)) {
            accepted = c;
        } else {
            double Z = 0.0;
            for (int j = lane; j < k; j += 32) {
                const double t = r[j] - w[j] * inv_s;
                w[j] = t > 0.0 ? t : 0.0;
                Z += w[j];
            }
            Z = warp_sum(Z) + st->sigma * st->p_off;
            if (Z > 1e-300) {
                const double inv_Z = 1.0 / Z;
                for (int j = lane; j < k; j += 32) r[j] = w[j] * inv_Z;
                st->sigma *= inv_Z;
            }
            __syncwarp();
        }
        taken |= 1ull << jc;
    }
    if (accepted >= 0 && emit) {
        if (lane == 0) {
            a.out_tok[(size_t)b * (K + 1) + st->nacc] = sg ? sg->ttok[accepted] : a.tree_tok[(size_t)b * N + accepted];
            a.path_node[(size_t)b * (K + 1) + st->nacc + 1] = accepted;
        }
        ++st->nacc;
    }
    return accepted;
}

// The same node with the slots' dependent chain cut to its minimum (k <= 32 candidates and <= 32 children; anything
// else, and weights that underflow, go to walk_node_seq).  Lane j holds candidate j (replicated over the warp when
// k < 32, so that a sum over the candidates is log2 k shuffle steps), lane i holds child i.
//   - What a slot's proposal is does not depend on the decisions before it: child i sees the candidates its earlier
//     siblings did not draw, q_i(j) = e_j / s_i with e_j = exp((c_j - max c)/T) and s_i the sum of the remaining e_j
//     (the same quotient as with the maximum of the remaining ones as reference).  All s_i at once, before the chain.
//   - The residual is carried unnormalised: r = rho / Zc.  A rejection gives rho_j <- max(rho_j - Zc q_i(j), 0) and
//     Zc <- sum_j rho_j + p_off, where p_off (the target's mass outside the candidates) stays what it was: dividing
//     by Zc gives back the normalised update, with sigma = 1 / Zc.  One fused multiply-add and one sum per slot.
//   - The acceptance test of child i needs rho at its own candidate and Zc as they were when the chain reached it;
//     lane i keeps them and all ratios are formed together after the chain, which runs over all children whether or
//     not an earlier one is accepted (the first accepted child decides; what follows it is ignored).
__device__ int walk_node(const WalkArgs &a, const Topo &topo, int b, int u, double M, double S, uint32_t thr, int lane,
                         WalkSmem *sm, WalkState *st, const WalkStage *sg = nullptr, bool emit = true) {
    const int k = a.k, N = a.N, K = a.K;
    // children of u, in slot order
    const int8_t *par = (sg && sg->parent) ? sg->parent : nullptr;  // (a lane-indexed read of the by-value struct is slow)
    const unsigned cm_lo = __ballot_sync(
        0xffffffffu, lane > u && lane < N && (par ? par[lane < N ? lane : 0] : topo.parent[lane < N ? lane : 0]) == u);
    const unsigned cm_hi = __ballot_sync(0xffffffffu, lane + 32 > u && lane + 32 < N &&
                                                          (par ? par[lane + 32 < N ? lane + 32 : 0]
                                                               : topo.parent[lane + 32 < N ? lane + 32 : 0]) == u);
    const int m_lo = __popc(cm_lo), m = m_lo + __popc(cm_hi);
    if (k > 32 || m > 32) return walk_node_seq(a, topo, b, u, M, S, thr, lane, sm, st, sg, emit);
    const int hd = topo.depth[u];
    int kp = 1;
    while (kp < k) kp <<= 1;
    const int j = lane & (kp - 1);
    const bool have = j < k;
    const double inv_T = 1.0 / a.T, inv_S = 1.0 / S;
    // the candidates: token, proposal weight, target probability
    const bool staged = sg && sg->e;
    double rho = 0.0, e = 0.0;
    if (staged) {
        if (have) {
            if (sg->p) {
                rho = sg->p[u * k + j];
            } else {
                const uint32_t bits = sg->pre[u * k + j];
                rho = ord_key(bits) >= thr ? exp(((double)bf16_bits_to_float((uint16_t)bits) - M) * inv_T) * inv_S : 0.0;
            }
            e = sg->e[hd * k + j];
            if (lane < k) sm->id[j] = sg->cid[hd * k + j];
        }
    } else {
        float clj = -INFINITY;
        if (have) {
            const int tok = sg ? sg->cid[hd * k + j] : SR_CHECKED(a.cand_id[((size_t)b * K + hd) * k + j], a.V, b);
            clj = sg ? sg->clog[hd * k + j] : a.cand_logit[((size_t)b * K + hd) * k + j];
            const uint32_t bits = sg ? sg->pre[u * k + j] : a.cand_target[((size_t)b * N + u) * k + j];
            const double l = (double)bf16_bits_to_float((uint16_t)bits);
            rho = ord_key(bits) >= thr ? exp((l - M) * inv_T) * inv_S : 0.0;
            if (lane < k) sm->id[j] = tok;
        }
        float mxf = clj;
        for (int o = kp >> 1; o > 0; o >>= 1) mxf = fmaxf(mxf, __shfl_xor_sync(0xffffffffu, mxf, o));
        e = have ? exp(((double)clj - (double)mxf) * inv_T) : 0.0;
    }
    double pc = rho;
    for (int o = kp >> 1; o > 0; o >>= 1) pc += __shfl_xor_sync(0xffffffffu, pc, o);
    const double p_off = pc < 1.0 ? 1.0 - pc : 0.0;
    // the children: lane i holds child i
    int c_i = 0, jc_i = 0;
    double uu_i = 0.0;
    if (lane < m) {
        c_i = lane < m_lo ? (int)__fns(cm_lo, 0, lane + 1) : 32 + (int)__fns(cm_hi, 0, lane - m_lo + 1);
        jc_i = SR_CHECKED((int)(sg ? sg->tcand[c_i] : a.tree_cand[(size_t)b * N + c_i]), k, b);
        uu_i = (double)(sg ? sg->uacc[c_i] : a.u_acc[(size_t)b * N + c_i]);
    }
    unsigned taken_i = lane < m ? (1u << jc_i) : 0u;  // exclusive prefix OR over the children before i
    {
        unsigned incl = taken_i;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl |= t;
        }
        taken_i = incl & ~taken_i;
    }
    double s_i = 0.0;
    if (staged) {
        for (int jj = 0; jj < k; ++jj)
            if (!((taken_i >> jj) & 1u)) s_i += sg->e[hd * k + jj];
    } else {
        for (int jj = 0; jj < k; ++jj) {
            const double ej = __shfl_sync(0xffffffffu, e, jj);
            if (!((taken_i >> jj) & 1u)) s_i += ej;
        }
    }
    if (__ballot_sync(0xffffffffu, lane < m && !(s_i > 0.0 && s_i < INFINITY)))
        return walk_node_seq(a, topo, b, u, M, S, thr, lane, sm, st, sg, emit);
    // what a slot needs from its child, where every lane can read it without a shuffle
    const double inv_s_i = lane < m ? 1.0 / s_i : 0.0;
    if (lane < m) {
        sm->inv_s[lane] = inv_s_i;
        sm->taken[lane] = taken_i;
        sm->jc[lane] = jc_i;
    }
    __syncwarp();
    // the chain
    double Zc = 1.0, my_rho = 0.0, my_Zc = 1.0;
    for (int i = 0; i < m; ++i) {
        const double q = ((sm->taken[i] >> j) & 1u) ? 0.0 : e * sm->inv_s[i];
        const double rho_jc = __shfl_sync(0xffffffffu, rho, sm->jc[i]);
        if (lane == i) {
            my_rho = rho_jc;
            my_Zc = Zc;
        }
        const double t = fmax(rho - Zc * q, 0.0);
        double Zn = t;
        for (int o = kp >> 1; o > 0; o >>= 1) Zn += __shfl_xor_sync(0xffffffffu, Zn, o);
        Zn += p_off;
        if (Zn > 1e-300 * Zc) {
            rho = t;
            Zc = Zn;
        }
    }
    // child i's own proposal probability: its candidate is among those it can still draw
    const double my_q = __shfl_sync(0xffffffffu, e, jc_i) * inv_s_i;
    // every child's test at once
    bool acc_i = false;
    float mg_i = INFINITY;
    if (lane < m) {
        double ratio;
        if (my_q > 0.0)
            ratio = my_rho > 0.0 ? (my_rho / my_Zc) / my_q : 0.0;
        else
            ratio = my_rho > 0.0 ? INFINITY : 0.0;
        acc_i = uu_i < (ratio < 1.0 ? ratio : 1.0);
        mg_i = (float)fabs(uu_i - ratio);
    }
    const unsigned accmask = __ballot_sync(0xffffffffu, acc_i);
    const int first = accmask ? __ffs(accmask) - 1 : -1;
    float mg = (lane < m && (first < 0 || lane <= first)) ? mg_i : INFINITY;
    mg = -warp_max(-mg);
    if (mg < st->mm) st->mm = mg;
    if (first >= 0) {
        const int accepted = __shfl_sync(0xffffffffu, c_i, first);
        if (emit) {
            if (lane == 0) {
                a.out_tok[(size_t)b * (K + 1) + st->nacc] = sg ? sg->ttok[accepted] : a.tree_tok[(size_t)b * N + accepted];
                a.path_node[(size_t)b * (K + 1) + st->nacc + 1] = accepted;
            }
            ++st->nacc;
        }
        return accepted;
    }
    // all rejected: the residual, normalised as the callers expect it (r and sigma = 1 / Zc)
    const double inv_Zc = 1.0 / Zc;
    if (lane < k) sm->r[j] = rho * inv_Zc;
    st->sigma = inv_Zc;
    st->p_off = p_off;
    __syncwarp();
    return -1;
}

// Results of a sequence and the hand-over of the residual (S = normaliser of u's row) to the terminal draw.
__device__ __forceinline__ void walk_end(const WalkArgs &a, int b, int u, double S, int lane, WalkSmem *sm,
                                         WalkState *st) {
    const int k = a.k;
    if (st->have_residual) {
        const double sigma = __shfl_sync(0xffffffffu, st->sigma, 0);
        const double f = S / sigma;  // (one division; the entries may be zero)
        for (int j = lane; j < k; j += 32) {
            a.ws_ovid[(size_t)b * k + j] = sm->id[j];
            a.ws_ovm[(size_t)b * k + j] = sm->r[j] * f;
        }
    }
    if (lane == 0) {
        a.ws_nov[b] = st->have_residual ? k : 0;
        a.n_acc[b] = st->nacc;
        a.term_node[b] = u;
        a.term_kind[b] = st->kind;
        if (a.min_margin) a.min_margin[b] = st->mm;
    }
}

// Bytes of shared memory the staged inputs of one sequence take (16-byte multiples per array).
__host__ __device__ inline size_t walk_stage_bytes(int N, int K, int k) {
    auto up = [](size_t x) { return (x + 15) / 16 * 16; };
    return 4 * up((size_t)N * 4) + up((size_t)N) + 2 * up((size_t)K * k * 4) + up((size_t)N * k * 2);
}

// The same for a CTA that examines nodes with all its warps: the parent array and the proposal weights too.
struct WalkBuf {
    float *rmax, *rsum, *uacc;
    int32_t *ttok;
    uint8_t *tcand;
    int32_t *cid;
    float *clog;
    uint16_t *pre;
    int8_t *parent;
    double *e;
};
__host__ __device__ inline size_t walk_buf_bytes(int N, int K, int k) {
    auto up = [](size_t x) { return (x + 15) / 16 * 16; };
    return walk_stage_bytes(N, K, k) + up((size_t)N) + up((size_t)K * k * sizeof(double));
}
__device__ __forceinline__ WalkBuf walk_buf(unsigned char *p, int N, int K, int k) {
    auto take = [&](size_t x) {
        unsigned char *q = p;
        p += (x + 15) / 16 * 16;
        return q;
    };
    WalkBuf w;
    w.rmax = reinterpret_cast<float *>(take((size_t)N * 4));
    w.rsum = reinterpret_cast<float *>(take((size_t)N * 4));
    w.uacc = reinterpret_cast<float *>(take((size_t)N * 4));
    w.ttok = reinterpret_cast<int32_t *>(take((size_t)N * 4));
    w.tcand = reinterpret_cast<uint8_t *>(take((size_t)N));
    w.cid = reinterpret_cast<int32_t *>(take((size_t)K * k * 4));
    w.clog = reinterpret_cast<float *>(take((size_t)K * k * 4));
    w.pre = reinterpret_cast<uint16_t *>(take((size_t)N * k * 2));
    w.parent = reinterpret_cast<int8_t *>(take((size_t)N));
    w.e = reinterpret_cast<double *>(take((size_t)K * k * sizeof(double)));
    return w;
}
// Fills everything but the row statistics, by all threads of a CTA; complete after the caller's next __syncthreads().
__device__ __forceinline__ void walk_buf_fetch(const WalkArgs &a, const Topo &topo, int b, const WalkBuf &w) {
    const int N = a.N, K = a.K, k = a.k, tid = threadIdx.x, nt = blockDim.x;
    for (int n = tid; n < N; n += nt) {
        w.uacc[n] = a.u_acc[(size_t)b * N + n];
        w.ttok[n] = a.tree_tok[(size_t)b * N + n];
        w.tcand[n] = a.tree_cand[(size_t)b * N + n];
        w.parent[n] = topo.parent[n];
    }
    for (int e = tid; e < K * k; e += nt) {
        w.cid[e] = SR_CHECKED(a.cand_id[(size_t)b * K * k + e], a.V, b);
        w.clog[e] = a.cand_logit[(size_t)b * K * k + e];
    }
    for (int e = tid; e < N * k; e += nt) {
        const int u = e / k, j = e - u * k;
        if (topo.n_child[u] > 0) {  // (a node with children is at depth < K)
            const int t = SR_CHECKED(a.cand_id[((size_t)b * K + topo.depth[u]) * k + j], a.V, b);
            w.pre[e] = a.logits ? a.logits[((size_t)b * N + u) * a.V + t] : a.cand_target[(size_t)b * N * k + e];
        }
    }
    // the proposal weights of every head's candidates, relative to the head's largest logit
    const double inv_T = 1.0 / a.T;
    __syncthreads();
    for (int e = tid; e < K * k; e += nt) {
        const int hd = e / k;
        float mx = -INFINITY;
        for (int jj = 0; jj < k; ++jj) mx = fmaxf(mx, w.clog[hd * k + jj]);
        w.e[e] = exp(((double)w.clog[e] - (double)mx) * inv_T);
    }
}

// The children of every node, grouped by parent in slot order, and what a slot's test needs of the proposal (k <= 32): known
// before the row statistics are.
struct WalkSlots {
    double *q;       // [N, k] the slot's proposal on the candidates: e_j / s over those the earlier siblings left, 0 on the others
    double *u;       // [N]    the acceptance uniform
    int32_t *node;   // [N]    the child
    int32_t *jc;     // [N]    its own candidate
    int32_t *start;  // [N]    first slot of a parent's children
};
__host__ __device__ inline size_t walk_slots_bytes(int N, int k) {
    auto up = [](size_t x) { return (x + 15) / 16 * 16; };
    return k > 32 ? 0 : up((size_t)N * k * sizeof(double)) + up((size_t)N * sizeof(double)) + 3 * up((size_t)N * sizeof(int32_t));
}
__device__ __forceinline__ WalkSlots walk_slots(unsigned char *p, int N, int k) {
    auto take = [&](size_t x) {
        unsigned char *q = p;
        p += (x + 15) / 16 * 16;
        return q;
    };
    WalkSlots w;
    w.q = reinterpret_cast<double *>(take((size_t)N * k * sizeof(double)));
    w.u = reinterpret_cast<double *>(take((size_t)N * sizeof(double)));
    w.node = reinterpret_cast<int32_t *>(take((size_t)N * sizeof(int32_t)));
    w.jc = reinterpret_cast<int32_t *>(take((size_t)N * sizeof(int32_t)));
    w.start = reinterpret_cast<int32_t *>(take((size_t)N * sizeof(int32_t)));
    return w;
}
// By all threads of a CTA, from a filled WalkBuf (a barrier before and after is the caller's).  *odd: set where a slot's weights
// underflow (such trees go through walk_node).
__device__ __forceinline__ void walk_slots_fill(const WalkBuf &buf, const Topo &topo, int N, int k, int where, const WalkSlots &w,
                                                int *odd) {
    // a thread per (child, candidate): the sums over the candidates are formed by each for itself, in the order walk_node has
    for (int e = threadIdx.x; e < (N - 1) * k; e += blockDim.x) {
        const int c = 1 + e / k, j = e - (c - 1) * k, u = buf.parent[c];
        int at = 0, first = 0;
        unsigned taken = 0u;
        for (int n = 1; n < N; ++n) {
            const int pn = buf.parent[n];
            at += pn < u || (pn == u && n < c);
            first += pn < u;
            if (pn == u && n < c) taken |= 1u << SR_CHECKED((int)buf.tcand[n], k, where);
        }
        const double *eh = buf.e + topo.depth[u] * k;
        double s = 0.0;
        for (int i = 0; i < k; ++i)
            if (!((taken >> i) & 1u)) s += eh[i];
        if (!(s > 0.0 && s < INFINITY)) *odd = 1;
        w.q[at * k + j] = ((taken >> j) & 1u) ? 0.0 : eh[j] * (1.0 / s);
        if (j == 0) {
            w.node[at] = c;
            w.jc[at] = SR_CHECKED((int)buf.tcand[c], k, where);
            w.u[at] = (double)buf.uacc[c];
            w.start[u] = first;
        }
    }
}

// One node by kp lanes (the power of two that holds k <= 32 candidates, and so all children; several nodes per warp, u < 0: a
// group without one): the arithmetic of walk_node with the slots' proposals ready.  rho: lane j's candidate's target
// probability, at the end its residual, not normalised.  Returns the accepted child or -1; mg: the smallest margin.
__device__ __forceinline__ int walk_group(const Topo &topo, int u, int k, int kp, double &rho, const WalkSlots &w, float &mg) {
    const int lane = threadIdx.x & 31, grp = lane / kp, j = lane & (kp - 1);
    const int m = u >= 0 ? topo.n_child[u] : 0, st = u >= 0 ? w.start[u] : 0;
    int most = m;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) most = max(most, __shfl_xor_sync(0xffffffffu, most, o));
    double pc = rho;
    for (int o = kp >> 1; o > 0; o >>= 1) pc += __shfl_xor_sync(0xffffffffu, pc, o);
    const double p_off = pc < 1.0 ? 1.0 - pc : 0.0;
    double Zc = 1.0, my_rho = 0.0, my_Zc = 1.0;
#pragma unroll 2
    for (int i = 0; i < most; ++i) {
        const bool on = i < m;
        const double q = on && j < k ? w.q[(st + i) * k + j] : 0.0;
        const double rho_jc = __shfl_sync(0xffffffffu, rho, on ? w.jc[st + i] : 0, kp);
        if (j == i) {
            my_rho = rho_jc;
            my_Zc = Zc;
        }
        const double t0 = rho - Zc * q, t = t0 > 0.0 ? t0 : 0.0;
        double Zn = t;
        for (int o = kp >> 1; o > 0; o >>= 1) Zn += __shfl_xor_sync(0xffffffffu, Zn, o);
        Zn += p_off;
        if (on && Zn > 1e-300 * Zc) {
            rho = t;
            Zc = Zn;
        }
    }
    // every child's test at once, lane i of the group child i
    bool acc = false;
    int c = -1;
    mg = INFINITY;
    if (j < m) {
        c = w.node[st + j];
        const double my_q = w.q[(st + j) * k + w.jc[st + j]], uu = w.u[st + j];
        double ratio;
        if (my_q > 0.0)
            ratio = my_rho > 0.0 ? (my_rho / my_Zc) / my_q : 0.0;
        else
            ratio = my_rho > 0.0 ? INFINITY : 0.0;
        acc = uu < (ratio < 1.0 ? ratio : 1.0);
        mg = (float)fabs(uu - ratio);
    }
    const unsigned mask = kp == 32 ? 0xffffffffu : ((1u << kp) - 1u) << (grp * kp);
    const unsigned hits = __ballot_sync(0xffffffffu, acc) & mask;
    const int f = hits ? __ffs(hits) - 1 : -1;
    if (f >= 0 && lane > f) mg = INFINITY;
    for (int o = kp >> 1; o > 0; o >>= 1) mg = fminf(mg, __shfl_xor_sync(0xffffffffu, mg, o));
    const int child = __shfl_sync(0xffffffffu, c, f >= 0 ? f : lane);
    return f < 0 ? -1 : child;
}

// The walk alone, one warp per sequence, on the target logits of the nodes' candidates (a.cand_target): read node by node.
__global__ void __launch_bounds__(WALK_WARPS * 32) walk_kernel(WalkArgs a, Topo topo) {
    __shared__ WalkSmem sh[WALK_WARPS];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int b = blockIdx.x * WALK_WARPS + warp;
    if (b >= a.B) return;
    WalkSmem *sm = &sh[warp];
    const float *row_max = a.row_max + (size_t)b * a.N, *row_sum = a.row_sum + (size_t)b * a.N;
    WalkState st;
    walk_begin(a, b, lane, &st);
    int u = 0;
    for (;;) {
        if (topo.n_child[u] == 0) {
            st.kind = (u != 0) ? 1 : 0;
            st.have_residual = false;
            break;
        }
        const int acc = walk_node(a, topo, b, u, (double)row_max[u], (double)row_sum[u], 0u, lane, sm, &st);
        if (acc < 0) {
            st.kind = 0;
            st.have_residual = true;
            break;
        }
        u = acc;
    }
    walk_end(a, b, u, (double)row_sum[u], lane, sm, &st);
}

// Maximum and sum of exponentials of one row by all NUC_THREADS threads of n_cta CTAs (a cluster; 1: a CTA alone); every
// thread returns with the result.  The row is cut into interleaved parts, a number that follows its length, and the parts
// are shared by the CTAs; a part's pairs (one per warp) and their sum are formed in one order however many CTAs there are, so
// that the result does not follow the batch size to the last bit (the thresholds and draws behind it would).  sm_ms:
// ROW_PARTS * NUC_THREADS / 32 pairs, at the same offset in every CTA (the caller has a cluster barrier between two rows).
constexpr int ROW_PARTS = 8;  // at most; the largest cluster
// The P parts from part0 on of n_parts: pairs of this warp to sm_ms[q * W + warp].  Vector j * NUC_THREADS + thread of the row
// belongs to part j % n_parts.  A thread takes up to R of a part's vectors together, which is what keeps R loads in flight: their
// maximum first, then the exponentials, which nothing rescales on the way.  The sums over the warp are formed for all parts
// at once, with the additions of warp_sum.  MORE: a part has more than R vectors per thread.  (Lazy verification, V 151936: 4
// sequences 37.4 -> 35.4 us, 256 sequences 105.5 -> 104.5 against sums in the order of the CTAs at hand; 256 of V 32000 38.4 ->
// 40.5, 200 of V 129000 93 -> 98.  A running pair per part, rescaled vector by vector and reduced part by part: 125 us for 105.5.)
template <int P, int R, bool MORE = false>
__device__ __forceinline__ void row_parts(const uint4 *__restrict__ p, int nvec, int part0, int n_parts, float c, float2 *sm_ms) {
    constexpr int W = NUC_THREADS / 32;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, step = NUC_THREADS * n_parts;
    auto as2 = [](uint32_t w) { return *reinterpret_cast<const __nv_bfloat162 *>(&w); };
    float m[P], s[P];
#pragma unroll
    for (int q = 0; q < P; ++q) {
        m[q] = NEG_INF;
        s[q] = 0.f;
#pragma unroll 1
        for (int i = (part0 + q) * NUC_THREADS + threadIdx.x; !MORE || i < nvec; i += R * step) {
            uint4 v[R];
#pragma unroll
            for (int r = 0; r < R; ++r) v[r] = ld_nc_v4(p + min(i + r * step, nvec - 1));
            __nv_bfloat162 m2 = as2(0xff80ff80u);  // (-inf, -inf)
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const __nv_bfloat162 x = __hmax2(__hmax2(as2(v[r].x), as2(v[r].y)), __hmax2(as2(v[r].z), as2(v[r].w)));
                if (i + r * step < nvec) m2 = __hmax2(m2, x);
            }
            const float mc = fmaxf(__low2float(m2), __high2float(m2));
            if (mc > m[q]) {
                s[q] *= ex2_approx((m[q] - mc) * c);  // (0 * 2^-inf = 0 at first)
                m[q] = mc;
            }
            const float nmc = m[q] == NEG_INF ? 0.f : -m[q] * c;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                if (i + r * step >= nvec) break;
                const uint32_t w[4] = {v[r].x, v[r].y, v[r].z, v[r].w};
                float acc = 0.f;
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    acc += ex2_approx(fmaf(__uint_as_float(w[t] << 16), c, nmc));
                    acc += ex2_approx(fmaf(__uint_as_float(w[t] & 0xffff0000u), c, nmc));
                }
                s[q] += acc;
            }
            if (!MORE) break;
        }
    }
    float mw[P];
#pragma unroll
    for (int q = 0; q < P; ++q) {
        mw[q] = warp_max_redux(m[q]);
        s[q] = m[q] == NEG_INF ? 0.f : s[q] * ex2_approx((m[q] - mw[q]) * c);
    }
    constexpr int L = P == 8 ? 3 : P == 4 ? 2 : P == 2 ? 1 : 0;
    const float sum = warp_sum_many<L>(s, lane);  // (of part lane >> (5 - L))
    float mine = mw[0];
#pragma unroll
    for (int q = 1; q < P; ++q)
        if (lane >> (5 - L) == q) mine = mw[q];
    if ((lane & ((1 << (5 - L)) - 1)) == 0) sm_ms[(lane >> (5 - L)) * W + warp] = make_float2(mine, sum);
}
__device__ void row_stats_row(const uint16_t *__restrict__ row_logits, int V, float c, float2 *sm_ms, int n_cta, int rank,
                              float *M_out, float *S_out) {
    constexpr int W = NUC_THREADS / 32;
    const uint4 *p = reinterpret_cast<const uint4 *>(row_logits);
    const int nvec = V >> 3, lane = threadIdx.x & 31;
    // so many parts that a thread has two to four vectors of each (more where the row has more than eight times that)
    const int lg = nvec > 8192 ? 3 : nvec > 4096 ? 2 : nvec > 2048 ? 1 : 0, n_parts = 1 << lg;
    const int P = n_parts > n_cta ? n_parts / n_cta : 1;  // per CTA; CTAs beyond the parts have none
    __syncthreads();
    if (nvec > 5 * ROW_PARTS * NUC_THREADS) {
        if (P == 8) row_parts<8, 5, true>(p, nvec, 0, 8, c, sm_ms);
        else if (P == 4) row_parts<4, 5, true>(p, nvec, rank * 4, 8, c, sm_ms);
        else if (P == 2) row_parts<2, 5, true>(p, nvec, rank * 2, 8, c, sm_ms);
        else row_parts<1, 5, true>(p, nvec, rank, 8, c, sm_ms);
    } else if (nvec > 4 * ROW_PARTS * NUC_THREADS) {
        if (P == 8) row_parts<8, 5>(p, nvec, 0, 8, c, sm_ms);
        else if (P == 4) row_parts<4, 5>(p, nvec, rank * 4, 8, c, sm_ms);
        else if (P == 2) row_parts<2, 5>(p, nvec, rank * 2, 8, c, sm_ms);
        else row_parts<1, 5>(p, nvec, rank, 8, c, sm_ms);
    } else {
        if (P == 8) row_parts<8, 4>(p, nvec, 0, 8, c, sm_ms);
        else if (P == 4) row_parts<4, 4>(p, nvec, rank * 4, n_parts, c, sm_ms);
        else if (P == 2) row_parts<2, 4>(p, nvec, rank * 2, n_parts, c, sm_ms);
        else if (rank < n_parts) row_parts<1, 4>(p, nvec, rank, n_parts, c, sm_ms);
    }
    if (n_cta > 1)
        cluster_sync_all();
    else
        __syncthreads();
    // every warp for itself: pair j of the row by lane j % 32, four pairs per lane
    float2 e[ROW_PARTS * W / 32];
    float mb = NEG_INF, sb = 0.f;
#pragma unroll
    for (int j = 0; j < ROW_PARTS * W / 32; ++j) {
        const int w = j * 32 + lane, part = w / W;
        e[j] = make_float2(NEG_INF, 0.f);
        if (part < n_parts) {
            const int r = part / P, at = w - r * P * W;
            if (n_cta == 1) {
                e[j] = sm_ms[at];
            } else {
                const double d = ld_dsmem_f64(sm_ms + at, r);
                e[j] = make_float2(__int_as_float(__double2loint(d)), __int_as_float(__double2hiint(d)));
            }
        }
        mb = fmaxf(mb, e[j].x);
    }
    mb = warp_max_redux(mb);
#pragma unroll
    for (int j = 0; j < ROW_PARTS * W / 32; ++j) sb += e[j].x == NEG_INF ? 0.f : e[j].y * ex2_approx((e[j].x - mb) * c);
    *M_out = mb;
    *S_out = warp_sum(sb);
}

// ------------------------------------------------------------------------------ terminal draw

struct TermArgs {
    const uint16_t *logits;
    const float *u_fin;
    const float *row_max;
    const int32_t *n_acc, *term_node;
    const int32_t *ws_nov, *ws_ovid;
    const double *ws_ovm;
    int32_t *out_tok;
    int32_t B, N, K, k, V;
    float c;  // log2(e) / T
};

// Plain softmax masses of eight tokens; tokens below the nucleus threshold (thr = 0: none) weigh nothing.
__device__ __forceinline__ void masses8(const uint4 &v, float M, float c, uint32_t thr, float (&e)[8]) {
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
    if (thr == 0u) {  // (uniform over the CTA) no truncation: nothing to compare, a third of the instructions
        const float nm = -M * c;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            e[2 * i] = ex2_approx(fmaf(__uint_as_float(w[i] << 16), c, nm));
            e[2 * i + 1] = ex2_approx(fmaf(__uint_as_float(w[i] & 0xffff0000u), c, nm));
        }
        return;
    }
    // the order of the keys is the order of the values (-0 = +0): compare two logits at a time with the
    // threshold's value
    const uint32_t tb = (thr & 0x8000u) ? (thr & 0x7fffu) : (~thr & 0xffffu);  // the key undone
    const uint32_t tb2 = tb | (tb << 16);
    const __nv_bfloat162 t2 = *reinterpret_cast<const __nv_bfloat162 *>(&tb2);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float e0 = ex2_approx(fmaf(__uint_as_float(w[i] << 16), c, -M * c));
        const float e1 = ex2_approx(fmaf(__uint_as_float(w[i] & 0xffff0000u), c, -M * c));
        const uint32_t keep = __hge2_mask(*reinterpret_cast<const __nv_bfloat162 *>(&w[i]), t2);
        e[2 * i] = (keep & 0xffffu) ? e0 : 0.f;
        e[2 * i + 1] = (keep >> 16) ? e1 : 0.f;
    }
}
__device__ __forceinline__ float mass1(uint16_t bits, float M, float c, uint32_t thr) {
    return ord_key(bits) >= thr ? ex2_approx(fmaf(bf16_bits_to_float(bits), c, -M * c)) : 0.f;  // same form as masses8
}

__device__ __forceinline__ double warp_incl_scan(double v, int lane) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        double t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += t;
    }
    return v;
}

// Pass 1 of the terminal draw by one warp: the plain softmax mass of every 32-vector slice of the segment
// [v_lo, v_hi) of a row, eight slices' loads in flight, left in out[0 .. n_sl).
__device__ __forceinline__ void term_slice_masses(const uint4 *__restrict__ p, int v_lo, int v_hi, int n_sl, float M, float c,
                                                  uint32_t thr, int lane, double *out) {
    // A slice's 256 masses are added pairwise in fp32 (relative error of a few 2^-24, the size of the exponentials' own
    // error); everything above a slice is fp64.  (Converting every mass to fp64 first kept the conversion pipe busy for
    // as long as the exponentials.)
    auto sum8 = [&](const uint4 &v) {
        float e[8];
        masses8(v, M, c, thr, e);
        return ((e[0] + e[1]) + (e[2] + e[3])) + ((e[4] + e[5]) + (e[6] + e[7]));
    };
    for (int s0 = 0; s0 < n_sl; s0 += 8) {
        uint4 v[8];  // (a load under a condition of its own ends up behind the use of the one before it: clamped instead)
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] = ld_nc_v4(p + max(0, min(v_lo + (s0 + q) * 32 + lane, v_hi - 1)));
        float x[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            x[q] = sum8(v[q]);
            if (v_lo + (s0 + q) * 32 + lane >= v_hi) x[q] = 0.f;
        }
        // eight sums over the warp at once: every step halves the values a lane carries (lane bits 4, 3, 2 pick the slice)
#pragma unroll
        for (int h = 4, o = 16; h > 0; h >>= 1, o >>= 1) {
            const bool up = lane & o;
#pragma unroll
            for (int q = 0; q < h; ++q) {
                const float give = up ? x[q] : x[q + h], keep = up ? x[q + h] : x[q];
                x[q] = keep + __shfl_xor_sync(0xffffffffu, give, o);
            }
        }
        x[0] += __shfl_xor_sync(0xffffffffu, x[0], 2);
        x[0] += __shfl_xor_sync(0xffffffffu, x[0], 1);
        if ((lane & 3) == 0 && s0 + (lane >> 2) < n_sl) out[s0 + (lane >> 2)] = (double)x[0];
    }
}

// The masses of the eight tokens of vector i of a row (zero beyond v_hi), the residual entries in place of the
// plain masses of their tokens; returns their sum.
__device__ __forceinline__ double term_vector_masses(const uint4 *__restrict__ p, int i, int v_hi, float M, float c, uint32_t thr,
                                                     int nov, const int32_t *ovid, const double *ovm, double (&ms)[8]) {
    double lsum = 0.0;
    if (i < v_hi) {
        float e[8];
        masses8(ld_nc_v4(p + i), M, c, thr, e);
#pragma unroll
        for (int t = 0; t < 8; ++t) ms[t] = (double)e[t];
        for (int j = 0; j < nov; ++j) {
            const int off = ovid[j] - i * 8;
            if (off >= 0 && off < 8) {
#pragma unroll
                for (int t = 0; t < 8; ++t)
                    if (t == off) ms[t] = ovm[j];
            }
        }
#pragma unroll
        for (int t = 0; t < 8; ++t) lsum += ms[t];
    } else {
#pragma unroll
        for (int t = 0; t < 8; ++t) ms[t] = 0.0;
    }
    return lsum;
}

// The token inside a 32-vector slice, by the warp whose lanes hold the vectors' masses (ms, their sums lsum): the
// first token whose running mass, from base on, exceeds the target; take_last: the last one with positive mass.
__device__ __forceinline__ void term_pick_token(int i, const double (&ms)[8], double lsum, double base, double target,
                                                bool take_last, int v_hi, int32_t *dst, int lane) {
    const double incl = warp_incl_scan(lsum, lane);
    const unsigned hit = take_last ? 0u : __ballot_sync(0xffffffffu, base + incl > target);
    if (hit) {
        const int Lh = __ffs(hit) - 1;
        if (lane == Lh) {
            int tok = -1;
            double cum = base + (incl - lsum);
#pragma unroll
            for (int t = 0; t < 8; ++t) {
                cum += ms[t];
                if (tok < 0 && cum > target) tok = i * 8 + t;
            }
            if (tok < 0) {  // scan and sequential sums disagreed in the last bit
#pragma unroll
                for (int t = 0; t < 8; ++t)
                    if (ms[t] > 0.0) tok = i * 8 + t;
            }
            *dst = tok;
        }
    } else {
        // the lanes' scanned mass fell short of the slice's sum by rounding: last token with positive mass
        int last_pos = -1;
#pragma unroll
        for (int t = 0; t < 8; ++t)
            if (ms[t] > 0.0) last_pos = i * 8 + t;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) last_pos = max(last_pos, __shfl_xor_sync(0xffffffffu, last_pos, o));
        if (lane == 0) *dst = last_pos < 0 ? max(0, v_hi * 8 - 1) : last_pos;
    }
}

// Last step of the terminal draw by one warp, inside the segment [v_lo, v_hi) that holds the target mass: seg_slices =
// the segment's n_sl slice masses (residual entries applied), base = the mass before the segment; ovid / ovm = the nov
// residual entries.  Writes the token to *dst.
__device__ void term_pick(const uint4 *__restrict__ p, const double *seg_slices, int n_sl, int v_lo, int v_hi, double base,
                          double target, float M, float c, uint32_t thr, int nov, const int32_t *ovid, const double *ovm,
                          int32_t *dst, int lane) {
    // the slice inside the selected segment: first one whose running mass exceeds the target; if rounding made
    // the slices fall short of the segment's own sum, the last slice with positive mass
    int sl_sel = -1, sl_pos = -1;
    double base_pos = 0.0;
    for (int c0 = 0; c0 < n_sl && sl_sel < 0; c0 += 32) {
        const double v = (c0 + lane < n_sl) ? seg_slices[c0 + lane] : 0.0;
        const double incl = warp_incl_scan(v, lane);
        const unsigned hit = __ballot_sync(0xffffffffu, base + incl > target);
        const unsigned pos = __ballot_sync(0xffffffffu, v > 0.0);
        if (pos) {
            const int lp = 31 - __clz(pos);
            sl_pos = c0 + lp;
            base_pos = base + __shfl_sync(0xffffffffu, incl - v, lp);
        }
        if (hit) {
            const int lh = __ffs(hit) - 1;
            sl_sel = c0 + lh;
            base += __shfl_sync(0xffffffffu, incl - v, lh);
        } else {
            base += __shfl_sync(0xffffffffu, incl, 31);
        }
    }
    bool take_last = false;
    if (sl_sel < 0) {
        if (sl_pos < 0) {  // no mass at all in the segment (cannot be selected with positive total; keep a valid token)
            if (lane == 0) *dst = max(0, v_hi * 8 - 1);
            return;
        }
        sl_sel = sl_pos;
        base = base_pos;
        take_last = true;
    }
    // the token inside the slice
    const int i = v_lo + sl_sel * 32 + lane;
    double ms[8];
    const double lsum = term_vector_masses(p, i, v_hi, M, c, thr, nov, ovid, ovm, ms);
    term_pick_token(i, ms, lsum, base, target, take_last, v_hi, dst, lane);
}

// The vectors [v_base, v_base + nvec_r) of a row are cut into one segment per warp of a CTA, each walked in slices of 32
// vectors (one per lane); the n_cta CTAs of a cluster (1: a CTA alone) share the slices of every segment.  Pass 1 (all warps,
// independent loads) leaves the mass of every slice in shared memory, those of the cluster's other CTAs are read by its first
// CTA; the residual entries (nov tokens ovid, masses ovm) then replace the plain mass of their tokens; two scans pick the segment
// and the slice that hold the target, and only that slice is read again to find the token.  Segments, slices and the order of all
// sums are the same however many CTAs there are: the draw from a flat tail follows their last bits.
//   thr       nucleus threshold key of the row, 0 for none
//   bits(j)   the bf16 logit of token ovid[j]
//   base      the mass before v_base; target < 0: u times the total
// By all TERM_THREADS threads of every CTA; slices: draw_smem_bytes, at the same offset in every CTA.  Bound by latency
// (a few hundred KB per sequence), which is why the loads of a round are issued together.
__host__ __device__ inline int draw_slices(int nvec) {
    const int vpw = (nvec + TERM_WARPS - 1) / TERM_WARPS;
    return ((vpw > 0 ? vpw : 1) + 31) / 32;
}
__host__ __device__ inline size_t draw_smem_bytes(int V) { return (size_t)TERM_WARPS * (draw_slices(V >> 3) + 1) * sizeof(double); }

template <class Bits>
__device__ void draw_row(const uint16_t *__restrict__ lg, int v_base, int nvec_r, float M, float c, uint32_t thr, int n_cta, int rank,
                         int nov, const int32_t *ovid, const double *ovm, Bits bits, double *slices, double base, double target,
                         float u, int32_t *dst) {
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint4 *p = reinterpret_cast<const uint4 *>(lg);
    constexpr int G = TERM_WARPS;
    const int vpw = (nvec_r + G - 1) / G > 0 ? (nvec_r + G - 1) / G : 1;  // vectors per segment
    const int n_sl = draw_slices(nvec_r);                                 // slices per segment
    const int per = (n_sl + n_cta - 1) / n_cta;                           // of them per CTA
    double *seg = slices + (size_t)G * n_sl;
    {
        const int v_lo = v_base + min(nvec_r, warp * vpw), v_hi = v_base + min(nvec_r, warp * vpw + vpw);
        const int s0 = min(n_sl, rank * per), s1 = min(n_sl, s0 + per);
        term_slice_masses(p, v_lo + s0 * 32, v_hi, s1 - s0, M, c, thr, lane, slices + (size_t)warp * n_sl + s0);
    }
    if (n_cta > 1) {
        cluster_sync_all();  // every CTA's slice masses are in its shared memory
        if (rank == 0)
            for (int e = tid; e < G * n_sl; e += TERM_THREADS) {
                const int r = e % n_sl / per;
                if (r > 0) slices[e] = ld_dsmem_f64(slices + e, r);
            }
        cluster_sync_all();  // the other CTAs may leave
        if (rank != 0) return;
    }
    __syncthreads();
    if (tid == 0) {
        for (int j = 0; j < nov; ++j) {
            const int vi = (ovid[j] >> 3) - v_base;
            if (vi < 0 || vi >= nvec_r) continue;  // (outside the vectors the draw works on)
            const int w = min(G - 1, vi / vpw), sl = (vi - w * vpw) >> 5;
            slices[w * n_sl + sl] += ovm[j] - (double)mass1(bits(j), M, c, thr);
        }
    }
    __syncthreads();
    {
        double acc = 0.0;
        for (int sl = lane; sl < n_sl; sl += 32) acc += slices[warp * n_sl + sl];
        acc = warp_sum(acc);
        if (lane == 0) seg[warp] = acc;
    }
    __syncthreads();
    if (warp != 0) return;
    const double v = lane < G ? seg[lane] : 0.0;
    if (target < 0.0) target = (double)u * warp_sum(v);
    const double incl = warp_incl_scan(v, lane);
    const unsigned hit = __ballot_sync(0xffffffffu, lane < G && base + incl > target);
    const int wsel = hit ? __ffs(hit) - 1 : -1;
    if (hit) base += __shfl_sync(0xffffffffu, incl - v, wsel);
    if (wsel < 0) {
        // the target reached the end of the masses through rounding: take the last token with positive mass (from the
        // end of the vectors the draw worked on, downwards)
        if (lane == 0) {
            int tok = (v_base + nvec_r) * 8 - 1;
            for (; tok > 0; --tok) {
                double ms = (double)mass1(lg[tok], M, c, thr);
                for (int j = 0; j < nov; ++j)
                    if (ovid[j] == tok) ms = ovm[j];
                if (ms > 0.0) break;
            }
            *dst = tok;
        }
        return;
    }
    const int v_lo = v_base + min(nvec_r, wsel * vpw), v_hi = v_base + min(nvec_r, wsel * vpw + vpw);
    term_pick(p, slices + (size_t)wsel * n_sl, n_sl, v_lo, v_hi, base, target, M, c, thr, nov, ovid, ovm, dst, lane);
}

// One CTA per sequence, for rows that were made after the walk (one per sequence).
__global__ void __launch_bounds__(TERM_THREADS) terminal_kernel(TermArgs a) {
    extern __shared__ double sh_slice[];
    const int b = blockIdx.x, nov = a.ws_nov[b];
    const uint16_t *lg = a.logits + (size_t)b * a.V;
    const int32_t *ovid = a.ws_ovid + (size_t)b * a.k;
    draw_row(lg, 0, a.V >> 3, a.row_max[(size_t)b * a.N + a.term_node[b]], a.c, 0u, 1, 0, nov, ovid, a.ws_ovm + (size_t)b * a.k,
             [&](int j) { return lg[ovid[j]]; }, sh_slice, 0.0, -1.0, a.u_fin[b], a.out_tok + (size_t)b * (a.K + 1) + a.n_acc[b]);
}

// ------------------------------------------------------------------------------ walk, a CTA per sequence

// One CTA per sequence, for the two variants in which something has to be computed per visited node before the
// node can be walked, and which nodes are visited is known only as the walk goes:
//   LAZY  the softmax statistics of a row are computed when the walk reaches it (at most K + 1 rows per
//         sequence instead of all N), and written to row_max / row_sum for those rows only;
//   NUC   the target distributions are their nuclei: the row's threshold is searched (nucleus_row) and left
//         in thr_key / keep_sum.
// Before each node all threads do that work, then warp 0 does the node.  The terminal draw from the last node's row,
// which the CTA has just read, follows in the same launch.
// A sequence's rows come one after the other and each waits for memory and shared-memory atomics, so a sequence gets a
// cluster of n_cta CTAs that share the passes over a row (walk_cta_split); the cluster's first CTA does the nodes.
struct WalkCtaLayout {
    size_t stage, slots, total;  // in front of the stage: the threshold search, whose place the draw's slice masses take
    bool grouped;                // a node by one group of lanes, with its slots' proposals (k <= 32, and where they fit: V < 5 M)
};
__host__ __device__ inline WalkCtaLayout walk_cta_layout(int N, int K, int k, int V, bool nuc) {
    WalkCtaLayout L;
    L.stage = draw_smem_bytes(V);
    if (nuc && L.stage < sizeof(NucleusSmem)) L.stage = sizeof(NucleusSmem);
    L.stage = (L.stage + 15) / 16 * 16;
    L.slots = L.stage + (walk_buf_bytes(N, K, k) + 15) / 16 * 16;
    L.grouped = k <= 32 && L.slots + walk_slots_bytes(N, k) <= (size_t)TERM_SMEM_LIMIT;
    L.total = L.slots + (L.grouped ? walk_slots_bytes(N, k) : 0);
    return L;
}

template <bool LAZY, bool NUC>
__global__ void __launch_bounds__(NUC_THREADS, 2)
walk_cta_kernel(WalkArgs a, Topo topo, float c, float top_p, float *__restrict__ row_max_w,
                float *__restrict__ row_sum_w, uint32_t *__restrict__ thr_key, float *__restrict__ keep_sum,
                float *__restrict__ out_thr, float *__restrict__ out_sum, int thr_ready, const float *__restrict__ u_fin,
                int n_cta) {
    extern __shared__ __align__(16) unsigned char nuc_raw[];
    NucleusSmem &nuc = *reinterpret_cast<NucleusSmem *>(nuc_raw);  // (NUC only)
    __shared__ WalkSmem sm;
    __shared__ float2 sm_ms[ROW_PARTS * NUC_THREADS / 32];
    __shared__ int sh_next[2];        // the next node, or -1 when the walk is over; rows in turn (one barrier per row)
    __shared__ uint32_t sh_last[4];   // of the last node, for the draw: threshold key, residual entries, accepted tokens
    __shared__ double sh_ovm[SPECROLL_MAX_TOPK];
    const int rank = n_cta > 1 ? (int)cluster_ctarank() : 0, b = blockIdx.x / n_cta;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    __shared__ int sh_odd;            // not grouped, or the slots' weights underflow: walk_node
    const WalkCtaLayout L = walk_cta_layout(a.N, a.K, a.k, a.V, NUC);
    const WalkBuf buf = walk_buf(nuc_raw + L.stage, a.N, a.K, a.k);
    const WalkSlots slots = walk_slots(nuc_raw + L.slots, a.N, a.k);
    const double inv_T = 1.0 / a.T;
    int kp = 1;
    while (kp < a.k) kp <<= 1;
    const WalkStage stage{buf.rmax, buf.rsum, buf.uacc, buf.ttok, buf.tcand, buf.cid, buf.clog, buf.pre, buf.parent, buf.e, nullptr};
    WalkState st;
    // Set up under the tail of the kernel before.  Where that is this call's own (statistics, thresholds), which itself
    // started when everything in front of the call was complete, the call's inputs are staged ahead of the wait.
    if (LAZY) pdl_wait();
    if (threadIdx.x == 0) sh_odd = !L.grouped;
    if (rank == 0) {
        walk_buf_fetch(a, topo, b, buf);
        __syncthreads();
        if (L.grouped) walk_slots_fill(buf, topo, a.N, a.k, b, slots, &sh_odd);
    }
    if (!LAZY) {
        pdl_wait();
        if (rank == 0)
            for (int n = threadIdx.x; n < a.N; n += NUC_THREADS) {
                buf.rmax[n] = a.row_max[(size_t)b * a.N + n];
                buf.rsum[n] = a.row_sum[(size_t)b * a.N + n];
            }
    }
    if (rank == 0 && warp == 0) walk_begin(a, b, lane, &st);
    __syncthreads();
    int u = 0;
    float M, S;
    for (int turn = 0;; turn ^= 1) {
        const size_t row = (size_t)b * a.N + u;
        const uint16_t *lg = a.logits + row * a.V;
        if constexpr (LAZY) {
            row_stats_row(lg, a.V, c, sm_ms, n_cta, rank, &M, &S);
            if (threadIdx.x == 0 && rank == 0) {
                row_max_w[row] = M;
                row_sum_w[row] = S;
            }
        } else {
            M = rank == 0 ? buf.rmax[u] : a.row_max[row];
            S = rank == 0 ? buf.rsum[u] : a.row_sum[row];
        }
        const bool search = NUC && !(thr_ready && topo.n_child[u] > 0);
        if (search) nucleus_row(lg, a.V, c, M, S, top_p, &nuc, n_cta, rank);
        if (rank == 0) {
            __syncthreads();  // (the staged inputs; the search's result)
            if (warp == 0) {
                uint32_t thr = 0u;
                float norm = S;
                if constexpr (NUC) {
                    thr = search ? nuc.prefix : thr_key[row];
                    norm = search ? nuc.keep : keep_sum[row];
                    if (lane == 0 && search) {
                        if (out_sum) out_sum[row] = norm;
                        if (out_thr) {  // the threshold as a logit: undo the key
                            const uint32_t bits = (thr & 0x8000u) ? (thr & 0x7fffu) : (~thr & 0xffffu);
                            out_thr[row] = __uint_as_float(bits << 16);
                        }
                    }
                }
                int next = -1;
                if (topo.n_child[u] == 0) {
                    st.kind = (u != 0) ? 1 : 0;
                    st.have_residual = false;
                } else if (!sh_odd) {
                    const bool mine = lane < a.k;  // (the first group of lanes has the node)
                    double rho = 0.0;
                    if (mine) {
                        const uint32_t bits = buf.pre[u * a.k + lane];
                        if (ord_key(bits) >= thr) rho = exp(((double)bf16_bits_to_float((uint16_t)bits) - (double)M) * inv_T) * (1.0 / (double)norm);
                    }
                    float mg;
                    next = __shfl_sync(0xffffffffu, walk_group(topo, lane < kp ? u : -1, a.k, kp, rho, slots, mg), 0);
                    st.mm = fminf(st.mm, __shfl_sync(0xffffffffu, mg, 0));
                    if (next >= 0) {
                        if (lane == 0) {
                            a.out_tok[(size_t)b * (a.K + 1) + st.nacc] = buf.ttok[next];
                            a.path_node[(size_t)b * (a.K + 1) + st.nacc + 1] = next;
                        }
                        ++st.nacc;
                    } else {
                        st.have_residual = true;
                        if (mine) sh_ovm[lane] = rho * (double)norm;  // (r = rho / Zc and sigma = 1 / Zc)
                    }
                } else {
                    next = walk_node(a, topo, b, u, (double)M, (double)norm, thr, lane, &sm, &st, &stage);
                    if (next < 0) st.have_residual = true;
                }
                if (next < 0 && st.have_residual && sh_odd) {
                    const double f = (double)norm / __shfl_sync(0xffffffffu, st.sigma, 0);  // (one division; the entries may be zero)
                    for (int j = lane; j < a.k; j += 32) sh_ovm[j] = sm.r[j] * f;
                }
                if (lane == 0) {
                    sh_next[turn] = next;
                    sh_last[0] = thr;
                    sh_last[1] = st.have_residual ? a.k : 0;
                    sh_last[2] = st.nacc;
                    if (next < 0) {
                        a.n_acc[b] = st.nacc;
                        a.term_node[b] = u;
                        a.term_kind[b] = st.kind;
                        if (a.min_margin) a.min_margin[b] = st.mm;
                    }
                }
            }
        }
        int next;
        if (n_cta > 1) {
            cluster_sync_all();
            next = (int)ld_dsmem_u32(&sh_next[turn], 0);
        } else {
            __syncthreads();
            next = sh_next[turn];
        }
        if (next < 0) break;
        u = next;
    }
    const uint32_t thr = n_cta > 1 ? ld_dsmem_u32(&sh_last[0], 0) : sh_last[0];
    draw_row(a.logits + ((size_t)b * a.N + u) * a.V, 0, a.V >> 3, M, c, thr, n_cta, rank, (int)sh_last[1],
             buf.cid + (sh_last[1] ? topo.depth[u] : 0) * a.k, sh_ovm, [&](int j) { return buf.pre[u * a.k + j]; },
             reinterpret_cast<double *>(nuc_raw), 0.0, -1.0, u_fin[b], a.out_tok + (size_t)b * (a.K + 1) + sh_last[2]);
}

// CTAs per row of walk_cta_kernel and nucleus_rows_kernel: as many as keep the grid within one wave of two CTAs per SM, a
// power of two up to the portable cluster size.  (Twice that, with a second wave: 128 sequences, V 151936, statistics of the
// visited rows 74 -> 98 us; the searches and nodes of a sequence wait for one another whatever their share of a row.)
constexpr int WALK_CTA_WAVE = 296;
static int walk_cta_split(int B) {
    int n = 8;
    while (n > 1 && (long long)B * n > WALK_CTA_WAVE) n >>= 1;
    return n;
}

// The nucleus thresholds of every node with children, one CTA per (sequence, such node), all at once: which of
// them the walk visits is not known yet, but a row's threshold depends on the row alone, and one pass of all
// of them over the machine costs less than the visited ones one after the other inside a sequence's walk.  (A
// sequence that ends at a leaf still needs that leaf's threshold for its last token: the walk kernel finds it.)
// A whole verification, us, walk alone -> thresholds ahead; rows = sequences x nodes with children:
//   V 151936, 8 such nodes:  32 rows 86 -> 73, 128: 99 -> 86, 256: 135 -> 127, 512: 155 -> 169, 768: 206 -> 240, 2048: 367 -> 475
//   V 152064, 22 such nodes: 88 rows 103 -> 90, 352: 140 -> 150, 704: 187 -> 225, 1408: 251 -> 354
//   V 32000, 8 such nodes:   32 rows 59 -> 53, 256: 67 -> 61, 512: 75 -> 78, 768: 85 -> 88, 2048: 105 -> 152
// The times cross near 300 rows, two per SM.  The line stays at five because up to there a call also leaves the thresholds and
// kept sums of the nodes with children that its walks do not visit.
#ifndef NUC_AHEAD_ROWS_PER_SM
#define NUC_AHEAD_ROWS_PER_SM 5
#endif
struct NodeList {
    int32_t n;
    int8_t node[SPECROLL_MAX_NODES];
};

__global__ void __launch_bounds__(NUC_THREADS, 2)
nucleus_rows_kernel(const uint16_t *__restrict__ logits, int V, int N, NodeList nodes, float c, float top_p,
                    const float *__restrict__ row_max, const float *__restrict__ row_sum,
                    uint32_t *__restrict__ thr_key, float *__restrict__ keep_sum, float *__restrict__ out_thr,
                    float *__restrict__ out_sum, int n_cta) {
    extern __shared__ __align__(16) unsigned char nuc_raw[];
    NucleusSmem &nuc = *reinterpret_cast<NucleusSmem *>(nuc_raw);
    pdl_wait();
    const int rank = n_cta > 1 ? (int)cluster_ctarank() : 0, r = blockIdx.x / n_cta;
    const int b = r / nodes.n, u = nodes.node[r - b * nodes.n];
    const size_t row = (size_t)b * N + u;
    const float M = row_max[row], S = row_sum[row];
    nucleus_row(logits + row * V, V, c, M, S, top_p, &nuc, n_cta, rank);
    if (n_cta > 1) cluster_sync_all();  // (the counts have been read)
    if (threadIdx.x == 0 && rank == 0) {
        const uint32_t thr = nuc.prefix;
        thr_key[row] = thr;
        keep_sum[row] = nuc.keep;
        if (out_sum) out_sum[row] = nuc.keep;
        if (out_thr) {  // the threshold as a logit: undo the key
            const uint32_t bits = (thr & 0x8000u) ? (thr & 0x7fffu) : (~thr & 0xffffu);
            out_thr[row] = __uint_as_float(bits << 16);
        }
    }
}

// ------------------------------------------------------------------------------ walk + terminal draw in one launch
//
// The plain verification after the row statistics, one cluster of S CTAs per sequence (S = 1: plain CTAs).
//   (1) Everything a walk can read is staged in shared memory; what does not depend on the row statistics (the
//       candidates, the uniforms, the target logits at the candidates) is fetched before the wait for the previous
//       kernel in the stream, which this kernel is launched to overlap with (programmatic dependent launch).
//   (2) Which nodes the walk reaches depends on its decisions, but what happens AT a node does not: its children
//       are tried in slot order until one is accepted, each against the residual left by the rejections before it.
//       So every node with children is examined on its own, all at once: the first accepted
//       child (or none, and then the residual), and the smallest margin on the way.  The walk itself is then a
//       chain of at most K + 1 look-ups.  Every CTA of a cluster does (1) and (2) for itself: same inputs, same
//       arithmetic, same result, nothing to exchange.
//   (3) The terminal draw over the last node's row: a warp of every CTA has one segment of the vocabulary, the CTAs of the
//       cluster share its slices; the slice masses of the other CTAs are read through distributed shared memory by the
//       cluster's first CTA, which finishes as terminal_kernel does.  (Letting the statistics pass leave the mass
//       of every slice of every row, so that this step reads a table and one slice, was tried: the table costs the
//       statistics kernel as much as it saves here.)
constexpr int WT_THREADS = TERM_THREADS;
constexpr int WT_SMEM_LIMIT = 160 * 1024;
constexpr int WT_WARPS = WT_THREADS / 32;
constexpr int TILE_STATIC_SMEM = 4 * 1024;                         // (at most) of the form without stored logits
constexpr int TILE_SMEM_LIMIT = 227 * 1024 - TILE_STATIC_SMEM;     // dynamic

// The nodes with children, in order, to par (by one warp); returns how many there are.  Ahead of the wait for the statistics: looked
// for node by node behind it, they were on the walk's critical path.
// Not where there are no stored logits: nothing of that kernel runs ahead of the projection's end, and a short walk takes longer with
// the list than it saves (1 sequence x 8 nodes 61.0 us, listed 64.3; 4 x 16 53.7 and 55.8; 32 x 32 106.7 and 107.2; 16 x 48 47.9 and 46.7).
__device__ __forceinline__ int walk_parents(const Topo &topo, int N, int8_t *par) {
    const int lane = threadIdx.x & 31;
    int n = 0;
    for (int u0 = 0; u0 < N; u0 += 32) {
        const bool inner = u0 + lane < N && topo.n_child[(u0 + lane) % SPECROLL_MAX_NODES] > 0;
        const unsigned mask = __ballot_sync(0xffffffffu, inner);
        if (inner) par[n + __popc(mask & ((1u << lane) - 1u))] = (int8_t)(u0 + lane);
        n += __popc(mask);
    }
    return n;
}

// Every node with children on its own.  first[u]: accepted child or -1, mm[u]: smallest margin, ovm[u, j]: the residual's
// masses where all children were rejected.  (A warp per node took 9 k
// cycles, two rounds of them where more than sixteen nodes have children: 10 us of the 66 us of 16 sequences x 48 nodes.)
// LISTED: par has the n_par nodes with children (walk_parents); else they are looked for here.
template <bool LISTED>
__device__ __forceinline__ void walk_nodes(const Topo &topo, int n_par, const int8_t *par, int k, const double *p, const float *rsum,
                                           const WalkSlots &w, int32_t *first, float *mm, double *ovm) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int kp = 1;
    while (kp < k) kp <<= 1;
    const int per_warp = 32 / kp, grp = lane / kp, j = lane & (kp - 1);
    if (!LISTED) {
        n_par = 0;
        for (int u = 0; u < topo.N; ++u) n_par += topo.n_child[u] > 0;
    }
    // as few nodes per warp as give every node a place in one round
    const int share = min(per_warp, (n_par + TERM_WARPS - 1) / TERM_WARPS);
    for (int i0 = warp * share; i0 < n_par; i0 += TERM_WARPS * share) {
        int u = -1;
        if (grp < share && i0 + grp < n_par) {
            if (LISTED) {
                u = par[i0 + grp];
            } else {
                int idx = 0;
                for (int n = 0; n < topo.N; ++n)
                    if (topo.n_child[n] > 0 && idx++ == i0 + grp) u = n;
            }
        }
        double rho = u >= 0 && j < k ? p[u * k + j] : 0.0;
        float mg;
        const int child = walk_group(topo, u, k, kp, rho, w, mg);
        if (u >= 0) {
            if (child < 0 && j < k) ovm[u * k + j] = rho * (double)rsum[u];  // (r = rho / Zc and sigma = 1 / Zc)
            if (j == 0) {
                first[u] = child;
                mm[u] = mg;
            }
        }
    }
}

struct WtLayout {
    size_t stage, ovm, first, mm, slices, p, slots, total;
    bool grouped;  // (as WalkCtaLayout's; V < 3 M)
};
__host__ __device__ inline WtLayout wt_layout(int N, int K, int k, size_t draw_bytes) {
    WtLayout L;
    auto up = [](size_t x) { return (x + 15) / 16 * 16; };
    size_t o = 0;
    L.stage = o;
    o += up(walk_buf_bytes(N, K, k));
    L.ovm = o;
    o += up((size_t)N * k * sizeof(double));
    L.first = o;
    o += up((size_t)N * sizeof(int32_t));
    L.mm = o;
    o += up((size_t)N * sizeof(float));
    L.slices = o;
    o += up(draw_bytes);
    L.p = o;
    o += up((size_t)N * k * sizeof(double));
    L.slots = o;
    L.grouped = k <= 32 && o + walk_slots_bytes(N, k) <= (size_t)WT_SMEM_LIMIT;
    if (L.grouped) o += up(walk_slots_bytes(N, k));
    L.total = o;
    return L;
}

// The terminal draw without the logits row: the masses of the row's vocabulary tiles are known (mass, per tile and row:
// maximum and sum), and the logits of the one tile that holds the target are made here, from the row's hidden state and 128
// rows of W (a few hundred KB to a MB; the storing projection, with all of W, took 178 us for 32 sequences of the 7B
// shape).  They are the projection's own logits to the bit: the same tensor operations over the same slices of the
// contraction, with the tokens as M and the hidden row as the first of N = 16.  (Sums of another order, in fp32 by all threads,
// rounded to the neighbouring bf16 value now and then, and the draw turned or the difference fell to the tile's last token.)
// Bound by the chain of the ring's slices, one CTA per sequence: 17 us more than such sums by a cluster of eight CTAs for 16
// sequences (210 -> 227 us with the projection of 8 nodes each), the same from 32 sequences on.  (Asking L2 for the whole tile
// first: no change.)
namespace dt {
constexpr int ROWS = 16, BK = 64, UMMA_K = 16, MAX_STAGES = 8, MIN_STAGES = 2;
constexpr int W_BYTES = HEAD_TILE * BK * 2, H_BYTES = ROWS * BK * 2, STAGE_BYTES = W_BYTES + H_BYTES;
constexpr int TMEM_COLS = 32;
}  // namespace dt
static_assert(dt::MIN_STAGES * dt::STAGE_BYTES >= WT_WARPS * (int)sizeof(WalkSmem), "the walk's scratch fits the ring");
struct TileArgs {
    CUtensorMap H, W;    // [B * N, d] in boxes of dt::ROWS rows, [V, d] in boxes of HEAD_TILE
    const float2 *mass;  // [tiles][B * N]
    int32_t d, rows, stages;
};

// By all threads of a CTA.  tok: HEAD_TILE doubles; ring: 1024-byte aligned, t.stages * dt::STAGE_BYTES.  bits(j): the bf16 logit of
// the residual's token j.  *dst is -1 where a bounded wait ran out.
template <class Bits>
__device__ void draw_tile(const TileArgs &t, size_t row, int V, float M, float c, int nov, const int32_t *ovid, const double *ovm,
                          Bits bits, double *tok, uint32_t ring, float u, int32_t *dst) {
    using namespace dt;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int n_tiles = (V + HEAD_TILE - 1) / HEAD_TILE;
    __shared__ double seg[TERM_WARPS], sh_base[2];
    __shared__ int sh_tile, sh_last;
    __shared__ __align__(8) unsigned long long bars[2 * MAX_STAGES + 1];
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int abort_flag;
    auto full_bar = [&](int s) { return smem_u32(&bars[s]); };
    auto empty_bar = [&](int s) { return smem_u32(&bars[MAX_STAGES + s]); };
    const uint32_t done_bar = smem_u32(&bars[2 * MAX_STAGES]);
    if (tid == 0) {
        for (int s = 0; s < t.stages; ++s) {
            mbar_init(full_bar(s), 1);
            mbar_init(empty_bar(s), 1);
        }
        mbar_init(done_bar, 1);
        abort_flag = 0;
        fence_mbar_init();
    }
    if (warp == 1) {
        tmem_alloc(smem_u32(&tmem_slot), TMEM_COLS);
        tmem_relinquish();
    }
    auto tile_mass = [&](int i) {
        const float2 e = t.mass[(size_t)i * t.rows + row];
        // (the tokens' exponents were formed with -m c rounded, as those of the tile at hand below are with -M c)
        double m = e.x == NEG_INF ? 0.0 : (double)e.y * exp2((double)(e.x * c) - (double)(M * c));
        for (int j = 0; j < nov; ++j)
            if (ovid[j] / HEAD_TILE == i) m += ovm[j] - (double)mass1(bits(j), M, c, 0u);
        return fmax(m, 0.0);  // (a tile whose mass was all in replaced tokens, after rounding)
    };
    // a run of tiles per warp, then the tile within the run
    const int per = (n_tiles + TERM_WARPS - 1) / TERM_WARPS;
    {
        double x = 0.0;
        for (int i = warp * per + lane; i < min(n_tiles, (warp + 1) * per); i += 32) x += tile_mass(i);
        x = warp_sum(x);
        if (lane == 0) seg[warp] = x;
    }
    fence_proxy_async();  // (the walk's scratch was in the ring's place)
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;
    if (warp == 0) {
        const double v = lane < TERM_WARPS ? seg[lane] : 0.0;
        double incl = warp_incl_scan(v, lane);
        const double target = (double)u * __shfl_sync(0xffffffffu, incl, 31);
        unsigned hit = __ballot_sync(0xffffffffu, incl > target), pos = __ballot_sync(0xffffffffu, v > 0.0);
        bool last = hit == 0u;  // (rounding: the last token with mass)
        const int w = hit ? __ffs(hit) - 1 : pos ? 31 - __clz(pos) : 0;
        double base = __shfl_sync(0xffffffffu, incl - v, w);
        int at = -1, at_pos = min(w * per, n_tiles - 1);
        double base_pos = base;
        for (int i0 = w * per; i0 < min(n_tiles, (w + 1) * per) && at < 0; i0 += 32) {
            const double x = i0 + lane < min(n_tiles, (w + 1) * per) ? tile_mass(i0 + lane) : 0.0;
            incl = warp_incl_scan(x, lane);
            hit = last ? 0u : __ballot_sync(0xffffffffu, base + incl > target);
            pos = __ballot_sync(0xffffffffu, x > 0.0);
            if (pos) {
                at_pos = i0 + 31 - __clz(pos);
                base_pos = base + __shfl_sync(0xffffffffu, incl - x, 31 - __clz(pos));
            }
            if (hit) {
                at = i0 + __ffs(hit) - 1;
                base += __shfl_sync(0xffffffffu, incl - x, __ffs(hit) - 1);
            } else {
                base += __shfl_sync(0xffffffffu, incl, 31);
            }
        }
        if (at < 0) {
            at = at_pos;
            base = base_pos;
            last = true;
        }
        if (lane == 0) {
            sh_tile = at;
            sh_last = last ? 1 : 0;
            sh_base[0] = base;
            sh_base[1] = target;
        }
    }
    __syncthreads();
    // the tile's logits: D[token, 0] = W[token, :] . hidden row
    const int v0 = sh_tile * HEAD_TILE, n_tok = min(HEAD_TILE, V - v0), KB = (t.d + BK - 1) / BK;
    if (warp == 0) {
        if (lane == 0) {
            int kb = 0;
            for (; kb < KB; ++kb) {
                const int s = kb % t.stages;
                if (!mbar_wait(empty_bar(s), ((uint32_t)(kb / t.stages) & 1u) ^ 1u, &abort_flag)) break;
                const uint32_t sw = ring + s * STAGE_BYTES;
                mbar_arrive_expect_tx(full_bar(s), STAGE_BYTES);
                tma_load_2d(sw, &t.W, kb * BK, v0, full_bar(s));
                tma_load_2d(sw + W_BYTES, &t.H, kb * BK, (int)row, full_bar(s));
            }
            if (kb < KB)  // aborting: let the copies already in flight land before the CTA goes away
                for (int q = max(0, kb - t.stages); q < kb; ++q) {
                    const unsigned long long t0 = globaltimer_ns();
                    while (!mbar_try_wait(full_bar(q % t.stages), (uint32_t)(q / t.stages) & 1u) && globaltimer_ns() - t0 < 100000000ull) {
                    }
                }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            constexpr uint32_t idesc = idesc_bf16(HEAD_TILE, ROWS, false, false);
            bool ok = true;
            for (int kb = 0; kb < KB && ok; ++kb) {
                const int s = kb % t.stages;
                ok = mbar_wait(full_bar(s), (uint32_t)(kb / t.stages) & 1u, &abort_flag);
                if (!ok) break;
                tc_fence_after();
                const uint32_t sw = ring + s * STAGE_BYTES;
                const uint64_t adesc = smem_desc_sw128(sw, 1024, 0), bdesc = smem_desc_sw128(sw + W_BYTES, 1024, 0);
#pragma unroll
                for (int kk = 0; kk < BK / UMMA_K; ++kk) umma_ss(tmem, adesc + 2u * kk, bdesc + 2u * kk, idesc, (kb | kk) != 0 ? 1u : 0u);
                umma_commit(empty_bar(s));
            }
            if (ok) umma_commit(done_bar);
        }
    } else if (warp < 6) {
        const int at = (warp & 3) * 32;  // the TMEM lanes this warp may read
        const bool ok = __all_sync(0xffffffffu, mbar_wait(done_bar, 0u, &abort_flag));
        tc_fence_after();
        if (ok) {
            uint32_t r[32];
            tmem_ld32(tmem + ((uint32_t)at << 16), r);
            tmem_ld_wait();
            tok[at + lane] = at + lane < n_tok ? (double)mass1(__bfloat16_as_ushort(__float2bfloat16_rn(__uint_as_float(r[0]))), M, c, 0u) : 0.0;
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc(tmem, TMEM_COLS);
    }
    if (warp != 0) return;
    if (abort_flag) {
        if (lane == 0) *dst = -1;
        return;
    }
    double ms[8], lsum = 0.0;
#pragma unroll
    for (int e = 0; e < 8; ++e) ms[e] = lane * 8 < HEAD_TILE ? tok[lane * 8 + e] : 0.0;
    for (int j = 0; j < nov; ++j) {
        const int off = lane * 8 < HEAD_TILE ? ovid[j] - v0 - lane * 8 : -1;
#pragma unroll
        for (int e = 0; e < 8; ++e)
            if (e == off) ms[e] = ovm[j];
    }
#pragma unroll
    for (int e = 0; e < 8; ++e) lsum += ms[e];
    term_pick_token(v0 / 8 + lane, ms, lsum, sh_base[0], sh_base[1], sh_last != 0, (v0 + n_tok) / 8, dst, lane);
}

// TILES: the target's numbers come from the projection (a.cand_target, tile.mass) and not from stored logits.
template <bool TILES>
__global__ void __launch_bounds__(WT_THREADS, 2) walk_term_kernel(WalkArgs a, Topo topo, const float *__restrict__ u_fin, float c,
                                                               int S, const float2 *__restrict__ run_tab, float *__restrict__ row_max_w,
                                                               float *__restrict__ row_sum_w, const __grid_constant__ TileArgs tile) {
    __shared__ WalkSmem sh_static[TILES ? 1 : WT_WARPS];
    extern __shared__ __align__(16) unsigned char sh_dyn[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rank = S > 1 ? (int)cluster_ctarank() : 0;
    const int b = blockIdx.x / S;
    const int N = a.N, K = a.K, k = a.k;
    const WtLayout L = wt_layout(N, K, k, TILES ? HEAD_TILE * sizeof(double) : draw_smem_bytes(a.V));
    const WalkBuf buf = walk_buf(sh_dyn + L.stage, N, K, k);
    float *rmax = buf.rmax, *rsum = buf.rsum;
    const int32_t *ttok = buf.ttok, *cid = buf.cid;
    const uint16_t *pre = buf.pre;
    double *ovm = reinterpret_cast<double *>(sh_dyn + L.ovm);
    int32_t *first = reinterpret_cast<int32_t *>(sh_dyn + L.first);
    float *mmin = reinterpret_cast<float *>(sh_dyn + L.mm);
    double *slices = reinterpret_cast<double *>(sh_dyn + L.slices);
    double *wp = reinterpret_cast<double *>(sh_dyn + L.p);
    const double inv_T = 1.0 / a.T;
    // scratch of nodes examined by a warp each (TILES: in the ring's place, which is not in use yet)
    WalkSmem *const sh = TILES ? reinterpret_cast<WalkSmem *>(sh_dyn + L.total) : sh_static;
    // (1) inputs of this call, none of them written by the kernel before this one where that is the call's own (the
    // statistics).  TILES: whatever the caller has put in front of the call may still be writing them.
    if (TILES) pdl_wait();
    const WalkSlots slots = walk_slots(sh_dyn + L.slots, N, k);
    __shared__ int sh_odd, sh_n_par;
    __shared__ int8_t sh_par[TILES ? 1 : SPECROLL_MAX_NODES];
    if (tid == 0) sh_odd = !L.grouped;
    if (!TILES && warp == WT_WARPS - 1) {  // (the last warp has the least to fetch)
        const int n = walk_parents(topo, N, sh_par);
        if (lane == 0) sh_n_par = n;
    }
    walk_buf_fetch(a, topo, b, buf);
    __syncthreads();
    if (L.grouped) walk_slots_fill(buf, topo, N, k, b, slots, &sh_odd);
    pdl_wait();  // the row statistics are complete from here on
    if (!TILES && run_tab) {
        // a row's statistics from its eight runs, eight lanes per row (N <= 64: one round; the result as row_stats_kernel's)
        static_assert(WT_THREADS / RS_WARPS >= SPECROLL_MAX_NODES, "all rows at once");
        const int n = tid / RS_WARPS;
        const float2 e = n < N ? run_tab[((size_t)b * N + n) * RS_WARPS + tid % RS_WARPS] : make_float2(NEG_INF, 0.f);
        float m = e.x;
#pragma unroll
        for (int o = RS_WARPS / 2; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        float s = e.x == NEG_INF ? 0.f : e.y * ex2_approx((e.x - m) * c);
#pragma unroll
        for (int o = RS_WARPS / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (n < N && tid % RS_WARPS == 0) {
            rmax[n] = m;
            rsum[n] = s;
            row_max_w[(size_t)b * N + n] = m;
            row_sum_w[(size_t)b * N + n] = s;
        }
    } else {
        for (int n = tid; n < N; n += WT_THREADS) {
            rmax[n] = a.row_max[(size_t)b * N + n];
            rsum[n] = a.row_sum[(size_t)b * N + n];
        }
    }
    __syncthreads();
    // the target probabilities of every walkable node's candidates
    for (int e = tid; e < N * k; e += WT_THREADS) {
        const int u = e / k;
        if (topo.n_child[u] > 0)
            wp[e] = exp(((double)bf16_bits_to_float(pre[e]) - (double)rmax[u]) * inv_T) * (1.0 / (double)rsum[u]);
    }
    __syncthreads();
    // (2) every node with children on its own
    if (!sh_odd) {
        walk_nodes<!TILES>(topo, sh_n_par, sh_par, k, wp, rsum, slots, first, mmin, ovm);
    } else {
        const WalkStage stage{rmax, rsum, buf.uacc, ttok, buf.tcand, cid, buf.clog, pre, buf.parent, buf.e, wp};
        int idx = 0;
        for (int u = 0; u < N; ++u) {
            if (topo.n_child[u] == 0) continue;
            if ((idx++ % WT_WARPS) != warp) continue;
            WalkState st;
            st.nacc = 0;
            st.kind = 0;
            st.sigma = 1.0;
            st.p_off = 0.0;
            st.mm = INFINITY;
            st.have_residual = false;
            const int acc = walk_node(a, topo, b, u, (double)rmax[u], (double)rsum[u], 0u, lane, &sh[warp], &st, &stage, false);
            if (acc < 0) {
                const double f = (double)rsum[u] / st.sigma;
                for (int j = lane; j < k; j += 32) ovm[u * k + j] = sh[warp].r[j] * f;
            }
            if (lane == 0) {
                first[u] = acc;
                mmin[u] = st.mm;
            }
            __syncwarp();
        }
    }
    __syncthreads();
    // the walk: every thread follows the same chain
    int u = 0, nacc = 0, kind = 0;
    bool resid = false;
    float mm = INFINITY;
    const bool writer = (rank == 0 && tid == 0);
    if (writer) {
        for (int i = 0; i <= K; ++i) a.path_node[(size_t)b * (K + 1) + i] = a.out_tok[(size_t)b * (K + 1) + i] = -1;
        a.path_node[(size_t)b * (K + 1)] = 0;
    }
    for (;;) {
        if (topo.n_child[u] == 0) {
            kind = (u != 0) ? 1 : 0;
            break;
        }
        mm = fminf(mm, mmin[u]);
        const int ch = first[u];
        if (ch < 0) {
            resid = true;
            break;
        }
        if (writer) {
            a.out_tok[(size_t)b * (K + 1) + nacc] = ttok[ch];
            a.path_node[(size_t)b * (K + 1) + nacc + 1] = ch;
        }
        ++nacc;
        u = ch;
    }
    if (writer) {
        a.n_acc[b] = nacc;
        a.term_node[b] = u;
        a.term_kind[b] = kind;
        if (a.min_margin) a.min_margin[b] = mm;
    }

    // (3) the terminal draw from row u: the residual (k entries over the plain masses) or the plain distribution
    const int nov = resid ? k : 0;
    const int32_t *ovid = cid + (resid ? topo.depth[u] : 0) * k;
    const double *ovm_u = ovm + u * k;
    const float M = rmax[u];
    if constexpr (TILES) {
        draw_tile(tile, (size_t)b * N + u, a.V, M, c, nov, ovid, ovm_u, [&](int j) { return pre[u * k + j]; }, slices,
                  (smem_u32(sh_dyn + L.total) + 1023u) & ~1023u, u_fin[b], a.out_tok + (size_t)b * (K + 1) + nacc);
        return;
    }
    const uint16_t *lg = a.logits + ((size_t)b * N + u) * a.V;
    const int nvec = a.V >> 3;
    // With the statistics kernel's table of the row's eight runs (run_tab; then S = 1): the run that holds the target
    // is found from the table and only that eighth of the row is read, cut into G segments like a whole row
    // otherwise.  v_base, nvec_r: the vectors the draw works on; base0: the mass before them.
    __shared__ int sh_run;
    __shared__ double sh_b0t[2];
    int v_base = 0, nvec_r = nvec;
    if (run_tab) {
        if (warp == 0) {
            const float2 e = lane < RS_WARPS ? run_tab[((size_t)b * N + u) * RS_WARPS + lane] : make_float2(-INFINITY, 0.f);
            double v = (lane < RS_WARPS && e.x != -INFINITY) ? (double)e.y * (double)ex2_approx((e.x - M) * c) : 0.0;
            for (int j = 0; j < nov; ++j)
                if (rs_run_of_vec(nvec, ovid[j] >> 3) == lane) v += ovm_u[j] - (double)mass1(pre[u * k + j], M, c, 0u);
            v = fmax(v, 0.0);  // (a run whose mass was all in overridden tokens, after rounding)
            const double incl = warp_incl_scan(v, lane);
            const double total = __shfl_sync(0xffffffffu, incl, 31);
            const double target = (double)u_fin[b] * total;
            const unsigned hit = __ballot_sync(0xffffffffu, lane < RS_WARPS && incl > target);
            const unsigned pos = __ballot_sync(0xffffffffu, v > 0.0);
            // (rounding kept the target at or above the total: the last run with mass; the draw inside it then ends
            // at its last token with mass)
            const int r = hit ? __ffs(hit) - 1 : (pos ? 31 - __clz(pos) : 0);
            const double b0 = __shfl_sync(0xffffffffu, incl - v, r);
            if (lane == 0) {
                sh_run = r;
                sh_b0t[0] = b0;
                sh_b0t[1] = target;
            }
        }
        __syncthreads();
        int v_end;
        rs_run(nvec, sh_run, &v_base, &v_end);
        nvec_r = v_end - v_base;
    }
    draw_row(lg, v_base, nvec_r, M, c, 0u, S, rank, nov, ovid, ovm_u, [&](int j) { return pre[u * k + j]; }, slices,
             run_tab ? sh_b0t[0] : 0.0, run_tab ? sh_b0t[1] : -1.0, u_fin[b], a.out_tok + (size_t)b * (K + 1) + nacc);
}

// S CTAs per sequence: as many as keep the grid within about two CTAs per SM, a power of two up to the portable
// cluster size.
static int walk_term_split(int B) {
    int S = 8;
    while (S > 1 && (long long)B * S > 296) S >>= 1;
    return S;
}

// Vocabularies whose slice masses one CTA can hold.
static bool draw_fits(int V) { return (size_t)TERM_WARPS * draw_slices(V >> 3) * sizeof(double) <= (size_t)TERM_SMEM_LIMIT; }

static int launch_terminal(const TermArgs &ta, cudaStream_t st) {
    if (!draw_fits(ta.V)) return SPECROLL_ELIMIT;
    const int rc = device_setup(reinterpret_cast<const void *>(terminal_kernel), WALK_CTA_SMEM, nullptr);
    if (rc != SPECROLL_OK) return rc;
    terminal_kernel<<<ta.B, TERM_THREADS, draw_smem_bytes(ta.V), st>>>(ta);
    SR_LAUNCH_CHECK();
    return SPECROLL_OK;
}

}  // namespace specroll

// ------------------------------------------------------------------------------ entry points

using namespace specroll;

static int check_verify_desc(const specroll_verify_desc *d) {
    if (!d || d->B < 0 || d->N < 1 || d->N > SPECROLL_MAX_NODES || d->K < 1 || d->K > SPECROLL_MAX_HEADS ||
        d->k < 1 || d->k > SPECROLL_MAX_TOPK || d->V < 8 || (d->V % 8) || d->k > d->V ||
        !(d->temperature > 0.f) || (d->flags & ~SPECROLL_VERIFY_LAZY_STATS) != 0)
        return SPECROLL_EINVAL;
    return SPECROLL_OK;
}

static size_t verify_ws_base(const specroll_verify_desc *d) {
    size_t B = (size_t)d->B, k = (size_t)d->k;
    return align_up(B * k * sizeof(double), 256) + align_up(B * k * sizeof(int32_t), 256) +
           align_up(B * sizeof(int32_t), 256) + 256;
}

// The statistics kernel's table of every row's eight runs (plain verification with all rows' statistics).
static size_t verify_ws_runs(const specroll_verify_desc *d) {
    return align_up((size_t)d->B * d->N * RS_WARPS * sizeof(float2), 256);
}

extern "C" size_t specroll_verify_workspace_bytes(const specroll_verify_desc *d) {
    if (check_verify_desc(d) != SPECROLL_OK) return 0;
    return verify_ws_base(d) + ((d->flags & SPECROLL_VERIFY_LAZY_STATS) ? 0 : verify_ws_runs(d));
}

extern "C" size_t specroll_verify_nucleus_workspace_bytes(const specroll_verify_desc *d) {
    if (check_verify_desc(d) != SPECROLL_OK) return 0;
    const size_t rows = (size_t)d->B * d->N;
    return verify_ws_base(d) + align_up(rows * sizeof(uint32_t), 256) + align_up(rows * sizeof(float), 256);
}

// top_p in (0, 1): the target distributions are their nuclei; otherwise the plain softmax.
static int run_verify(const specroll_verify_desc *d, float top_p, const void *logits, const int32_t *parent_host,
                      const int32_t *tree_tok, const uint8_t *tree_cand, const int32_t *cand_id,
                      const float *cand_logit, const float *u_acc, const float *u_fin, int32_t *n_acc,
                      int32_t *path_node, int32_t *out_tok, int32_t *term_node, int32_t *term_kind, float *row_max,
                      float *row_sum, float *min_margin, float *nucleus_thr, float *nucleus_sum, void *workspace,
                      size_t workspace_bytes, void *cuda_stream, bool runs_optional = false) {
    if (check_verify_desc(d) != SPECROLL_OK) return SPECROLL_EINVAL;
    const bool truncate = top_p > 0.f && top_p < 1.f;
    Topo topo;
    if (build_topo(parent_host, d->N, d->K, d->k, &topo, nullptr) != SPECROLL_OK) return SPECROLL_EINVAL;
    if (d->B == 0) return SPECROLL_OK;  // (an empty batch has empty arrays: their pointers may be NULL)
    if (!logits || !tree_tok || !tree_cand || !cand_id || !cand_logit || !u_acc || !u_fin || !n_acc ||
        !path_node || !out_tok || !term_node || !term_kind || !row_max || !row_sum)
        return SPECROLL_EINVAL;
    if (!aligned16(logits)) return SPECROLL_EALIGN;
    const bool lazy = (d->flags & SPECROLL_VERIFY_LAZY_STATS) != 0;
    // the table of the rows' runs serves the plain verification with all rows' statistics; a caller with a fixed
    // scratch, or with the nucleus form's workspace, goes without it when it does not fit (the terminal draw then
    // reads the whole row, spread over a cluster for small batches)
    bool use_runs = !truncate && !lazy;
    if (use_runs && runs_optional && workspace_bytes < verify_ws_base(d) + verify_ws_runs(d)) use_runs = false;
    const size_t need = truncate ? specroll_verify_nucleus_workspace_bytes(d)
                                 : verify_ws_base(d) + (use_runs ? verify_ws_runs(d) : 0);
    if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255u) || workspace_bytes < need)
        return SPECROLL_EWORKSPACE;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    // (the workspace begins with the hand-over area of the walk on its own, which these kernels do not need)
    char *ws = static_cast<char *>(workspace) + verify_ws_base(d);
    const size_t n_rows = (size_t)d->B * d->N;
    uint32_t *thr_key = truncate ? reinterpret_cast<uint32_t *>(ws) : nullptr;
    float *keep_sum = truncate ? reinterpret_cast<float *>(ws + align_up(n_rows * sizeof(uint32_t), 256)) : nullptr;

    const float c = (float)(1.4426950408889634 / (double)d->temperature);
    const int rows = d->B * d->N;
    float2 *run_tab = use_runs ? reinterpret_cast<float2 *>(ws) : nullptr;  // (behind the hand-over area; no nucleus arrays in this form)
    int n_sm = 0;
    const int rc_sm = device_setup(nullptr, 0, &n_sm);
    if (rc_sm != SPECROLL_OK) return rc_sm;
    if (use_runs) {
        // Up to 44 runs per SM (814 rows) the form with the rings; with more rows there are warps enough, and the ring's
        // bookkeeping costs issue slots.  A whole verification, us, CTA per row -> rings:
        //   V 151936: 512 rows 47.2 -> 45.1, 768: 61.3 -> 61.0, 896: 66.6 -> 65.9, 1024: 68.0 -> 71.9, 1536: 95.6 -> 101.3
        //   V 64000:  512 rows 26.8 -> 25.9, 768: 34.0 -> 34.2, 896: 36.1 -> 36.9, 1024: 37.5 -> 39.5, 1536: 47.3 -> 51.6
        //   V 32000:  512 rows 21.3 -> 19.7, 768: 24.0 -> 23.1, 1024: 26.9 -> 26.0, 1536: 31.8 -> 37.2
        //   V 8000:   512 rows 18.8 -> 16.2, 1024: 20.3 -> 17.8, 1536: 21.6 -> 19.5
        // (20 rows of 152 k tokens from HBM 29 -> 19, 4096 rows 198 -> 234.)
        // With more than 38 runs per SM a warp for each of them, 44 warps per SM with two copies in flight, instead of 21 or so
        // with two runs each: too few warps keep the exponentials, the integer instructions and the waits apart.  21 warps -> 44:
        //   V 152064: 640 rows 50.1 -> 51.5, 768: 60.0 -> 58.4, 800: 62.1 -> 58.6;  V 64000: 640 28.0 -> 29.7, 768 35.3 -> 33.1, 800 34.7 -> 33.2
        const int n_runs = rows * RS_WARPS;
        // Not where a run is less than a group (V 8192) and most are empty: 800 rows of V 1024 14.9 -> 16.8, 2048 15.7 -> 14.8, 4096 14.8 ->
        // 15.3, 8000 15.6 -> 16.0.
        const bool more = n_runs > 38 * n_sm && d->V >= RS_WARPS * RUN_PIECE * 8;
        const int ctas = more ? RUN_CTAS_MORE : RUN_CTAS, most = RUN_WARPS * ctas * n_sm, rounds = (n_runs + most - 1) / most;
        if (n_runs <= 44 * n_sm) {
            // every warp the same number of runs (to one), and a CTA for each while there is room
            const int warps = (n_runs + rounds - 1) / rounds, grid = warps <= ctas * n_sm ? warps : ctas * n_sm;
            const int per_sm = (grid + n_sm - 1) / n_sm, piece_bytes = RUN_WARPS * RUN_PIECE * (int)sizeof(uint4);
            int ring_n = 200 * 1024 / per_sm / piece_bytes;
            ring_n = ring_n < RUN_RING_MIN ? RUN_RING_MIN : ring_n > RUN_RING_MAX ? RUN_RING_MAX : ring_n;
            auto *const kern = more ? run_stats_kernel<false, RUN_CTAS_MORE> : run_stats_kernel<false, RUN_CTAS>;
            const int rc_ = device_setup(reinterpret_cast<const void *>(kern), RUN_RING_MAX * piece_bytes, nullptr);
            if (rc_ != SPECROLL_OK) return rc_;
            SR_CUDA_TRY(launch_dependent(true, kern, dim3((unsigned)grid), dim3(32 * RUN_WARPS),
                                         (size_t)ring_n * piece_bytes, st, static_cast<const uint16_t *>(logits), d->V, c, n_runs, ring_n,
                                         run_tab, (float *)nullptr, (float *)nullptr));
        } else {
            SR_CUDA_TRY(launch_dependent(true, row_stats_kernel, dim3((unsigned)rows), dim3(RS_THREADS), 0, st,
                                         static_cast<const uint16_t *>(logits), d->V, c, (float *)nullptr, (float *)nullptr, run_tab));
        }
    } else if (!lazy) {
        // up to four rows per SM by the form with the rings (20 rows of 152 k tokens 19 -> 8 us), more by a CTA per row
        const int per_sm = (rows + n_sm - 1) / n_sm, piece_bytes = RS_WARPS * RUN_PIECE * (int)sizeof(uint4);
        if (per_sm <= 4) {
            int ring_n = 200 * 1024 / per_sm / piece_bytes;
            if (ring_n > RUN_RING_MAX) ring_n = RUN_RING_MAX;
            const int rc_ = device_setup(reinterpret_cast<const void *>(run_stats_kernel<true, 4>), RUN_RING_MAX * piece_bytes, nullptr);
            if (rc_ != SPECROLL_OK) return rc_;
            SR_CUDA_TRY(launch_dependent(true, run_stats_kernel<true, 4>, dim3((unsigned)rows), dim3(RS_THREADS), (size_t)ring_n * piece_bytes,
                                         st, static_cast<const uint16_t *>(logits), d->V, c, rows * RS_WARPS, ring_n, (float2 *)nullptr,
                                         row_max, row_sum));
        } else {
            SR_CUDA_TRY(launch_dependent(true, row_stats_kernel, dim3((unsigned)rows), dim3(RS_THREADS), 0, st,
                                         static_cast<const uint16_t *>(logits), d->V, c, row_max, row_sum, (float2 *)nullptr));
        }
    }

    WalkArgs wa;
    wa.logits = static_cast<const uint16_t *>(logits);
    wa.cand_target = nullptr;
    wa.tree_tok = tree_tok;
    wa.tree_cand = tree_cand;
    wa.cand_id = cand_id;
    wa.cand_logit = cand_logit;
    wa.u_acc = u_acc;
    wa.row_max = row_max;
    wa.row_sum = row_sum;
    wa.n_acc = n_acc;
    wa.path_node = path_node;
    wa.out_tok = out_tok;
    wa.term_node = term_node;
    wa.term_kind = term_kind;
    wa.min_margin = min_margin;
    wa.ws_nov = nullptr;
    wa.ws_ovid = nullptr;
    wa.ws_ovm = nullptr;
    wa.B = d->B;
    wa.N = d->N;
    wa.K = d->K;
    wa.k = d->k;
    wa.V = d->V;
    wa.T = (double)d->temperature;
    if (truncate || lazy) {
        const int n_cta = walk_cta_split(d->B);
        const size_t smem = walk_cta_layout(d->N, d->K, d->k, d->V, truncate).total;
        if (!draw_fits(d->V) || smem > (size_t)WALK_CTA_SMEM) return SPECROLL_ELIMIT;
        auto *const kern = truncate ? (lazy ? walk_cta_kernel<true, true> : walk_cta_kernel<false, true>) : walk_cta_kernel<true, false>;
        int rc_ = device_setup(reinterpret_cast<const void *>(kern), WALK_CTA_SMEM, nullptr);
        if (rc_ != SPECROLL_OK) return rc_;
        bool ahead = false;
        if (truncate && !lazy) {
            NodeList nodes;
            nodes.n = 0;
            for (int u = 0; u < d->N; ++u)
                if (topo.n_child[u] > 0) nodes.node[nodes.n++] = (int8_t)u;
            // Worth it while those rows are few enough to be searched side by side (small batches, whose walks
            // would otherwise search three or four rows one after the other on a nearly empty machine); with
            // more rows than that, searching only the visited ones inside the walk is less work and faster.
            int n_sm = 0;
            rc_ = device_setup(reinterpret_cast<const void *>(nucleus_rows_kernel), (int)sizeof(NucleusSmem), &n_sm);
            if (rc_ != SPECROLL_OK) return rc_;
            ahead = nodes.n > 0 && d->B * nodes.n <= NUC_AHEAD_ROWS_PER_SM * n_sm;
            if (ahead) {
                const int rows_cta = walk_cta_split(d->B * nodes.n);
                SR_CUDA_TRY(launch_clusters(true, rows_cta, nucleus_rows_kernel, dim3((unsigned)(d->B * nodes.n * rows_cta)),
                                            dim3(NUC_THREADS), sizeof(NucleusSmem), st, static_cast<const uint16_t *>(logits), d->V,
                                            d->N, nodes, c, top_p, row_max, row_sum, thr_key, keep_sum, nucleus_thr, nucleus_sum,
                                            rows_cta));
            }
        }
        SR_CUDA_TRY(launch_clusters(true, n_cta, kern, dim3((unsigned)(d->B * n_cta)), dim3(NUC_THREADS), smem, st, wa, topo, c,
                                    truncate ? top_p : 1.0f, row_max, row_sum, thr_key, keep_sum, truncate ? nucleus_thr : nullptr,
                                    truncate ? nucleus_sum : nullptr, ahead ? 1 : 0, u_fin, n_cta));
        return SPECROLL_OK;
    }
    // plain verification: the walk and the terminal draw in one launch, overlapping the statistics kernel's tail
    const int S = use_runs ? 1 : walk_term_split(d->B);
    const WtLayout L = wt_layout(d->N, d->K, d->k, draw_smem_bytes(d->V));
    if (L.total > (size_t)WT_SMEM_LIMIT) return SPECROLL_ELIMIT;
    const int rc_ = device_setup(reinterpret_cast<const void *>(walk_term_kernel<false>), WT_SMEM_LIMIT, nullptr);
    if (rc_ != SPECROLL_OK) return rc_;
    SR_CUDA_TRY(launch_clusters(true, S, walk_term_kernel<false>, dim3((unsigned)(d->B * S)), dim3(WT_THREADS), L.total, st, wa, topo,
                                u_fin, c, S, (const float2 *)run_tab, row_max, row_sum, TileArgs{}));
    return SPECROLL_OK;
}

// The hand-over area between the walk and the terminal draw inside a workspace (the layout of run_verify).
static void carve_verify_ws(const specroll_verify_desc *d, void *workspace, double **ovm, int32_t **ovid, int32_t **nov) {
    const size_t B = (size_t)d->B, k = (size_t)d->k;
    char *ws = static_cast<char *>(workspace);
    *ovm = reinterpret_cast<double *>(ws);
    ws += align_up(B * k * sizeof(double), 256);
    *ovid = reinterpret_cast<int32_t *>(ws);
    ws += align_up(B * k * sizeof(int32_t), 256);
    *nov = reinterpret_cast<int32_t *>(ws);
}

namespace specroll {
// want_id[(b, u), j] = cand_id[b, depth(u), j]: the tokens whose target logit the walk reads at node u
__global__ void want_ids_kernel(Topo topo, int B, int N, int K, int k, const int32_t *__restrict__ cand_id,
                                int32_t *__restrict__ want_id) {
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (size_t)B * N * k) return;
    const int j = (int)(i % k), u = (int)((i / k) % N), b = (int)(i / ((size_t)k * N));
    const int hd = min((int)topo.depth[u], K - 1);  // (a node of the last level has no children; any valid token)
    want_id[i] = cand_id[((size_t)b * K + hd) * k + j];
}
}  // namespace specroll

extern "C" int specroll_verify_want_ids(const specroll_verify_desc *d, const int32_t *parent_host,
                                        const int32_t *cand_id, int32_t *want_id, void *cuda_stream) {
    if (check_verify_desc(d) != SPECROLL_OK || !cand_id || !want_id) return SPECROLL_EINVAL;
    Topo topo;
    if (build_topo(parent_host, d->N, d->K, d->k, &topo, nullptr) != SPECROLL_OK) return SPECROLL_EINVAL;
    const size_t n = (size_t)d->B * d->N * d->k;
    if (n == 0) return SPECROLL_OK;
    want_ids_kernel<<<(unsigned)((n + 255) / 256), 256, 0, static_cast<cudaStream_t>(cuda_stream)>>>(
        topo, d->B, d->N, d->K, d->k, cand_id, want_id);
    SR_LAUNCH_CHECK();
    return SPECROLL_OK;
}

extern "C" int specroll_verify_walk_sparse(const specroll_verify_desc *d, const void *cand_target,
                                           const float *row_max, const float *row_sum, const int32_t *parent_host,
                                           const int32_t *tree_tok, const uint8_t *tree_cand, const int32_t *cand_id,
                                           const float *cand_logit, const float *u_acc, int32_t *n_acc,
                                           int32_t *path_node, int32_t *out_tok, int32_t *term_node,
                                           int32_t *term_kind, float *min_margin, void *workspace,
                                           size_t workspace_bytes, void *cuda_stream) {
    if (check_verify_desc(d) != SPECROLL_OK || d->flags != 0) return SPECROLL_EINVAL;
    Topo topo;
    if (build_topo(parent_host, d->N, d->K, d->k, &topo, nullptr) != SPECROLL_OK) return SPECROLL_EINVAL;
    if (d->B == 0) return SPECROLL_OK;  // (an empty batch has empty arrays: their pointers may be NULL)
    if (!cand_target || !row_max || !row_sum || !tree_tok || !tree_cand || !cand_id || !cand_logit || !u_acc || !n_acc ||
        !path_node || !out_tok || !term_node || !term_kind)
        return SPECROLL_EINVAL;
    if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255u) || workspace_bytes < verify_ws_base(d))
        return SPECROLL_EWORKSPACE;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    WalkArgs wa;
    wa.logits = nullptr;
    wa.cand_target = static_cast<const uint16_t *>(cand_target);
    wa.tree_tok = tree_tok;
    wa.tree_cand = tree_cand;
    wa.cand_id = cand_id;
    wa.cand_logit = cand_logit;
    wa.u_acc = u_acc;
    wa.row_max = row_max;
    wa.row_sum = row_sum;
    wa.n_acc = n_acc;
    wa.path_node = path_node;
    wa.out_tok = out_tok;
    wa.term_node = term_node;
    wa.term_kind = term_kind;
    wa.min_margin = min_margin;
    carve_verify_ws(d, workspace, &wa.ws_ovm, &wa.ws_ovid, &wa.ws_nov);
    wa.B = d->B;
    wa.N = d->N;
    wa.K = d->K;
    wa.k = d->k;
    wa.V = d->V;
    wa.T = (double)d->temperature;
    walk_kernel<<<(d->B + WALK_WARPS - 1) / WALK_WARPS, WALK_WARPS * 32, 0, st>>>(wa, topo);
    SR_LAUNCH_CHECK();
    return SPECROLL_OK;
}

extern "C" int specroll_verify_hidden(const specroll_verify_desc *d, int32_t dim, const void *hidden, const void *W,
                                      const void *cand_target, const void *tile_mass, const float *row_max, const float *row_sum,
                                      const int32_t *parent_host, const int32_t *tree_tok, const uint8_t *tree_cand,
                                      const int32_t *cand_id, const float *cand_logit, const float *u_acc, const float *u_fin,
                                      int32_t *n_acc, int32_t *path_node, int32_t *out_tok, int32_t *term_node, int32_t *term_kind,
                                      float *min_margin, void *cuda_stream) {
    if (check_verify_desc(d) != SPECROLL_OK || d->flags != 0 || dim < 8 || (dim % 8)) return SPECROLL_EINVAL;
    Topo topo;
    if (build_topo(parent_host, d->N, d->K, d->k, &topo, nullptr) != SPECROLL_OK) return SPECROLL_EINVAL;
    if (d->B == 0) return SPECROLL_OK;  // (an empty batch has empty arrays: their pointers may be NULL)
    if (!hidden || !W || !cand_target || !tile_mass || !row_max || !row_sum || !tree_tok || !tree_cand || !cand_id || !cand_logit ||
        !u_acc || !u_fin || !n_acc || !path_node || !out_tok || !term_node || !term_kind)
        return SPECROLL_EINVAL;
    if (!aligned16(hidden) || !aligned16(W) || (reinterpret_cast<uintptr_t>(tile_mass) & 7u)) return SPECROLL_EALIGN;
    WalkArgs wa;
    wa.logits = nullptr;
    wa.cand_target = static_cast<const uint16_t *>(cand_target);
    wa.tree_tok = tree_tok;
    wa.tree_cand = tree_cand;
    wa.cand_id = cand_id;
    wa.cand_logit = cand_logit;
    wa.u_acc = u_acc;
    wa.row_max = row_max;
    wa.row_sum = row_sum;
    wa.n_acc = n_acc;
    wa.path_node = path_node;
    wa.out_tok = out_tok;
    wa.term_node = term_node;
    wa.term_kind = term_kind;
    wa.min_margin = min_margin;
    wa.ws_nov = nullptr;
    wa.ws_ovid = nullptr;
    wa.ws_ovm = nullptr;
    wa.B = d->B;
    wa.N = d->N;
    wa.K = d->K;
    wa.k = d->k;
    wa.V = d->V;
    wa.T = (double)d->temperature;
    const WtLayout L = wt_layout(d->N, d->K, d->k, HEAD_TILE * sizeof(double));
    int n_sm = 0;
    int rc = device_setup(reinterpret_cast<const void *>(walk_term_kernel<true>), TILE_SMEM_LIMIT, &n_sm);
    if (rc != SPECROLL_OK) return rc;
    // a ring as deep as fits beside the walk, with room for a second CTA on an SM where there are more sequences than SMs
    TileArgs tile;
    const int room = (d->B > n_sm ? TILE_SMEM_LIMIT / 2 - TILE_STATIC_SMEM / 2 - 1024 : TILE_SMEM_LIMIT) - (int)L.total - 1024;
    tile.stages = std::max(dt::MIN_STAGES, std::min(dt::MAX_STAGES, room / dt::STAGE_BYTES));
    const size_t smem = L.total + 1024 + (size_t)tile.stages * dt::STAGE_BYTES;
    if (smem > (size_t)TILE_SMEM_LIMIT) return SPECROLL_ELIMIT;
    tile.mass = static_cast<const float2 *>(tile_mass);
    tile.d = dim;
    tile.rows = d->B * d->N;
    if ((rc = make_tmap_2d_bf16(&tile.H, hidden, (uint64_t)tile.rows, (uint64_t)dim, (uint64_t)dim, dt::ROWS)) != SPECROLL_OK) return rc;
    if ((rc = make_tmap_2d_bf16(&tile.W, W, (uint64_t)d->V, (uint64_t)dim, (uint64_t)dim, HEAD_TILE)) != SPECROLL_OK) return rc;
    SR_CUDA_TRY(launch_dependent(true, walk_term_kernel<true>, dim3((unsigned)d->B), dim3(WT_THREADS), smem,
                                 static_cast<cudaStream_t>(cuda_stream), wa, topo, u_fin, (float)(1.4426950408889634 / (double)d->temperature),
                                 1, (const float2 *)nullptr, (float *)nullptr, (float *)nullptr, tile));
    return SPECROLL_OK;
}

extern "C" int specroll_verify_terminal_rows(const specroll_verify_desc *d, const void *term_logits,
                                             const float *row_max, const int32_t *n_acc, const int32_t *term_node,
                                             const float *u_fin, int32_t *out_tok, void *workspace,
                                             size_t workspace_bytes, void *cuda_stream) {
    if (check_verify_desc(d) != SPECROLL_OK || d->flags != 0) return SPECROLL_EINVAL;
    if (d->B == 0) return SPECROLL_OK;  // (an empty batch has empty arrays: their pointers may be NULL)
    if (!term_logits || !row_max || !n_acc || !term_node || !u_fin || !out_tok) return SPECROLL_EINVAL;
    if (!aligned16(term_logits)) return SPECROLL_EALIGN;
    if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255u) || workspace_bytes < verify_ws_base(d))
        return SPECROLL_EWORKSPACE;
    TermArgs ta;
    double *ovm;
    int32_t *ovid, *nov;
    carve_verify_ws(d, workspace, &ovm, &ovid, &nov);
    ta.logits = static_cast<const uint16_t *>(term_logits);
    ta.u_fin = u_fin;
    ta.row_max = row_max;
    ta.n_acc = n_acc;
    ta.term_node = term_node;
    ta.ws_nov = nov;
    ta.ws_ovid = ovid;
    ta.ws_ovm = ovm;
    ta.out_tok = out_tok;
    ta.B = d->B;
    ta.N = d->N;
    ta.K = d->K;
    ta.k = d->k;
    ta.V = d->V;
    ta.c = (float)(1.4426950408889634 / (double)d->temperature);
    return launch_terminal(ta, static_cast<cudaStream_t>(cuda_stream));
}

extern "C" int specroll_verify(const specroll_verify_desc *d, const void *logits,
                               const int32_t *parent_host, const int32_t *tree_tok,
                               const uint8_t *tree_cand, const int32_t *cand_id,
                               const float *cand_logit, const float *u_acc, const float *u_fin,
                               int32_t *n_acc, int32_t *path_node, int32_t *out_tok,
                               int32_t *term_node, int32_t *term_kind, float *row_max,
                               float *row_sum, float *min_margin, void *workspace,
                               size_t workspace_bytes, void *cuda_stream) {
    return run_verify(d, 1.0f, logits, parent_host, tree_tok, tree_cand, cand_id, cand_logit, u_acc, u_fin, n_acc,
                      path_node, out_tok, term_node, term_kind, row_max, row_sum, min_margin, nullptr, nullptr,
                      workspace, workspace_bytes, cuda_stream);
}

extern "C" int specroll_verify_nucleus(const specroll_verify_desc *d, float top_p, const void *logits,
                                       const int32_t *parent_host, const int32_t *tree_tok,
                                       const uint8_t *tree_cand, const int32_t *cand_id,
                                       const float *cand_logit, const float *u_acc, const float *u_fin,
                                       int32_t *n_acc, int32_t *path_node, int32_t *out_tok,
                                       int32_t *term_node, int32_t *term_kind, float *row_max,
                                       float *row_sum, float *min_margin, float *nucleus_thr,
                                       float *nucleus_sum, void *workspace, size_t workspace_bytes,
                                       void *cuda_stream) {
    if (!(top_p > 0.f)) return SPECROLL_EINVAL;
    return run_verify(d, top_p, logits, parent_host, tree_tok, tree_cand, cand_id, cand_logit, u_acc, u_fin, n_acc,
                      path_node, out_tok, term_node, term_kind, row_max, row_sum, min_margin, nucleus_thr,
                      nucleus_sum, workspace, workspace_bytes, cuda_stream, /*runs_optional=*/true);
}

// ------------------------------------------------------------------------------ allocation-free variant
//
// Scratch of specroll_verify_static: lives in the library image, one copy per GPU that loads the
// library, held until the process exits.  Layout = the workspace layout of specroll_verify for the
// largest admitted problem (SPECROLL_STATIC_MAX_B sequences, SPECROLL_STATIC_MAX_BK residual entries).
namespace specroll {
constexpr size_t STATIC_SCRATCH_BYTES =
    (SPECROLL_STATIC_MAX_BK * sizeof(double) + 255) / 256 * 256 +
    (SPECROLL_STATIC_MAX_BK * sizeof(int32_t) + 255) / 256 * 256 +
    (SPECROLL_STATIC_MAX_B * sizeof(int32_t) + 255) / 256 * 256 + 256;
static __device__ __align__(256) unsigned char g_verify_scratch[STATIC_SCRATCH_BYTES];

constexpr int MAX_DEVICES = 64;
static void *g_scratch_addr[MAX_DEVICES];  // device address of g_verify_scratch, per device ordinal
static std::mutex g_scratch_mutex;
}  // namespace specroll

extern "C" int specroll_verify_static(const specroll_verify_desc *d, const void *logits,
                                      const int32_t *parent_host, const int32_t *tree_tok,
                                      const uint8_t *tree_cand, const int32_t *cand_id,
                                      const float *cand_logit, const float *u_acc, const float *u_fin,
                                      int32_t *n_acc, int32_t *path_node, int32_t *out_tok,
                                      int32_t *term_node, int32_t *term_kind, float *row_max,
                                      float *row_sum, float *min_margin, void *cuda_stream) {
    if (check_verify_desc(d) != SPECROLL_OK) return SPECROLL_EINVAL;
    if (d->B > SPECROLL_STATIC_MAX_B || (long long)d->B * d->k > SPECROLL_STATIC_MAX_BK) return SPECROLL_ELIMIT;
    if (verify_ws_base(d) > STATIC_SCRATCH_BYTES) return SPECROLL_ELIMIT;
    int dev = -1;
    SR_CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= MAX_DEVICES) return SPECROLL_ELIMIT;
    void *scratch = nullptr;
    {
        // In host code the array's name is only a handle; the kernels need its device address,
        // which differs per GPU.  Looked up once per device, with that device current.
        std::lock_guard<std::mutex> lock(g_scratch_mutex);
        if (!g_scratch_addr[dev]) {
            void *p = nullptr;
            SR_CUDA_TRY(cudaGetSymbolAddress(&p, g_verify_scratch));
            g_scratch_addr[dev] = p;
        }
        scratch = g_scratch_addr[dev];
    }
    // (the table of the rows' runs is used when it fits the scratch beside the hand-over area, else the terminal draw
    // reads the whole row)
    return run_verify(d, 1.0f, logits, parent_host, tree_tok, tree_cand, cand_id, cand_logit, u_acc, u_fin, n_acc,
                      path_node, out_tok, term_node, term_kind, row_max, row_sum, min_margin, nullptr, nullptr, scratch,
                      STATIC_SCRATCH_BYTES, cuda_stream, /*runs_optional=*/true);
}
