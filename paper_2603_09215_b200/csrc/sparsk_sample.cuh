// Nucleus (top-p) sampling with temperature over the id range of each sequence's modality
// (Sec. V-A: the 28-layer backbone decodes with temperature 0.7, top_p 0.9; the other backbone
// greedily, which is the arg max the heads already produce).
//
// No sort.  With w_i = exp((z_i - max z) / T):
//   1. the nucleus is every id whose w exceeds a threshold t, plus the first k ids (by id) whose
//      w equals t, where t is the largest value with  sum{w >= t} >= top_p * sum{w};
//   2. the drawn id is the one at which the cumulative mass, taken in decreasing w (equal w: lower
//      id first), first exceeds u * (kept mass); it has the largest w = v with sum{w >= v} > u * kept,
//      and among the ids with that w it is number floor((u * kept - sum{w > v}) / v).
// Both thresholds are found on the bit patterns of the positive floats (their unsigned order is
// their numeric order), four bits per pass: a pass sums the mass of the sixteen buckets that extend
// the prefix found so far.
//
// A row is read from memory once: every thread keeps its (up to 48) weights in registers for all
// passes, ids in order (CTA, thread, register).  A pass adds each weight into the thread's
// own column of a [16][512] shared-memory table (no conflicts, no atomics, a fixed order), the
// warps reduce the table, and, for ranges that need more than one CTA, the eight CTAs of a
// thread-block cluster combine their sixteen sums through distributed shared memory with one
// cluster barrier.  Ranges of up to 24,576 ids (the speech ranges) take one CTA per sequence,
// larger ones (the text ranges) a cluster of eight.  The uniform number u is the caller's (no
// generator on the device).
//
// Bound by instruction issue and barriers of the passes, not by bytes (a row is in the L2), so what
// counts is what a pass issues: 512 threads, because the table a pass clears and reduces is as
// wide as the CTA; only the registers that hold weights; the maximum, the total and the second
// search's first pass not as passes of their own.  A row of 6,561 ids 45.9 -> 20.5 us (16 registers a
// thread; 22.6 with room for 48, 26.7 with 1,024 threads of 24), of 16,384 57.4 -> 38.9 (1,024: 38.6),
// of 151,936 77.9 -> 53.3 (55.3), 64 of those 366 -> 245 (258).  It was 1,024 threads of 24.
#pragma once

#include <cooperative_groups.h>

#include "sparsk_common.cuh"

namespace sparsk {

namespace cg = cooperative_groups;

constexpr int SP_CLUSTER = 8;
constexpr int SP_STEP = 4;  // a loop over the weights ends at a multiple of this
constexpr int SP_THREADS = 512;
constexpr int SP_SHORT_REGS = 16, SP_REGS = 48;             // weights a thread holds (ranges of up to 8,192 ids; others)
constexpr int SP_CTA_RANGE = SP_THREADS * SP_REGS;          // ids one CTA holds: 24,576
constexpr int SP_MAX_RANGE = SP_CLUSTER * SP_CTA_RANGE;     // ids per modality: 196,608

struct SampleArgs {
    const float *logits;         // [n][V]; only the modality's range of a row is read
    const float *uniforms;       // [n] in [0, 1)
    const int *modality;         // [n]: 0 text ids [0, Vt), else speech ids [Vt, Vt + Vs)
    unsigned long long *key_out; // optional [n]: the drawn id in the arg max key format
    int *token_out;              // optional [n]
    int V, Vt, Vs;
    int only_modality;           // rows of the other modality are left to another launch
    float inv_temperature, top_p;
};

struct SampleShared {
    float part[2][16];  // this CTA's sums of a pass, read by the whole cluster; double buffered
    float bcast[16], top[16];
    float warp_x[32];
    int i[32];
    int cnt_part, before_cta, all_eq;
};

// One value per thread combined over the CTA and then over the cluster (sum, or max when MAX) in a
// fixed order; every thread gets the result.  `round` counts the calls of this and of combine16.
template <int CL, int T, bool MAX>
__device__ __forceinline__ float combine1(float x, SampleShared *sh, uint32_t &round)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, buf = round++ & 1;
    const float none = MAX ? -INFINITY : 0.f;
    x = MAX ? warp_max(x) : warp_sum(x);
    if (lane == 0) sh->warp_x[warp] = x;
    __syncthreads();
    x = lane < T / 32 ? sh->warp_x[lane] : none;
    x = MAX ? warp_max(x) : warp_sum(x);
    if (CL > 1) {
        cg::cluster_group cluster = cg::this_cluster();
        if (threadIdx.x == 0) sh->part[buf][0] = x;
        cluster.sync();
        x = lane < CL ? cluster.map_shared_rank(&sh->part[buf][0], lane)[0] : none;
        x = MAX ? warp_max(x) : warp_sum(x);
    }
    __syncthreads();  // warp_x is free again
    return x;
}

// Sums the table's sixteen rows (one value per thread each) over the CTA and then over the cluster
// in a fixed order; the sums are left in sh->bcast.  The caller has filled its column
// tab[c * T + tid].
template <int CL, int T>
__device__ __forceinline__ void combine16(float *tab, SampleShared *sh, uint32_t &round)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, buf = round++ & 1;
    __syncthreads();
    static_assert(T >= 512, "a warp per row of the table");
    if (warp < 16) {  // warp c combines row c: T / 32 values per lane, then across the lanes
        const float *row = tab + warp * T;
        float x = row[lane];
#pragma unroll
        for (int i = 1; i < T / 32; i++) x += row[i * 32 + lane];
        x = warp_sum(x);
        if (lane == 0) (CL > 1 ? sh->part[buf][warp] : sh->bcast[warp]) = x;
    }
    if (CL > 1) {
        cg::cluster_group cluster = cg::this_cluster();
        cluster.sync();  // also a barrier of this CTA
        if (warp < 16) {
            float x = 0.f;
            if (lane < CL) x = cluster.map_shared_rank(&sh->part[buf][0], lane)[warp];
            x = warp_sum(x);
            if (lane == 0) sh->bcast[warp] = x;
        }
    }
    __syncthreads();
    // the table and bcast are next written after barriers that every thread must reach first
}

// Largest bit pattern t with  mass{w >= t} >= target  (strict = false)  or  > target  (strict = true);
// `above` returns mass{w > t}, `at` returns mass{w == t}.
// The sums of the first pass (the weights by their top four bits) are the same in both searches of a
// row: `again` takes them from the search before.
template <int CL, int T, int REGS>
__device__ __forceinline__ uint32_t threshold_search(float *tab, const float (&w)[REGS], int per_thread, float target,
                                                     bool strict, bool again, float &above, float &at,
                                                     SampleShared *sh, uint32_t &round)
{
    uint32_t prefix = 0;
    float hi_mass = 0.f, bucket = 0.f;
    float *col = tab + threadIdx.x;
    for (int shift = 28; shift >= 0; shift -= 4) {
        const bool first = shift == 28;
        if (!(first && again)) {
#pragma unroll
            for (int c = 0; c < 16; c++) col[c * T] = 0.f;  // (its last readers are behind a barrier)
            const uint32_t want = first ? 0u : (prefix >> (shift + 4));
#pragma unroll
            for (int j = 0; j < REGS; j++) {
                if (j % SP_STEP == 0 && j >= per_thread) break;  // (weights past a thread's ids are zero)
                const uint32_t b = __float_as_uint(w[j]);
                if (first || (b >> (shift + 4)) == want) col[((b >> shift) & 15u) * T] += w[j];
            }
            combine16<CL, T>(tab, sh, round);
            if (first && threadIdx.x < 16) sh->top[threadIdx.x] = sh->bcast[threadIdx.x];  // (read much later)
        }
        const float *acc = first && again ? sh->top : sh->bcast;
        // the highest bucket whose mass, with everything above it, passes the target
        float v[16];
#pragma unroll
        for (int c = 0; c < 16; c++) v[c] = acc[c];
        int pick = 0;
        float run = hi_mass;
#pragma unroll
        for (int c = 15; c >= 1; c--) {
            const float with = run + v[c];
            if (strict ? with > target : with >= target) {
                pick = c;
                break;
            }
            run = with;
        }
        hi_mass = run;
        bucket = acc[pick];
        prefix |= (uint32_t)pick << shift;
    }
    above = hi_mass;
    at = bucket;
    return prefix;
}

// grid = n sequences x CL CTAs (cluster dimension CL when CL > 1); dynamic shared memory 16 * T * 4 bytes.
template <int CL, int T, int REGS>
__global__ void __launch_bounds__(T, 1) nucleus_sample_kernel(SampleArgs a)
{
    extern __shared__ __align__(16) float sp_tab[];
    __shared__ SampleShared sh;
    griddep_wait();
    const int b = blockIdx.x / CL, rank = blockIdx.x % CL, tid = threadIdx.x;
    const int mod = a.modality[b] != 0;
    if (a.only_modality >= 0 && mod != a.only_modality) return;  // uniform over the cluster
    const int lo = mod ? a.Vt : 0, n = mod ? a.Vs : a.Vt;
    const float *z = a.logits + (size_t)b * a.V + lo;
    if (n < 1 || n > CL * T * REGS) {
        if (rank == 0 && tid == 0 && a.token_out) a.token_out[b] = -1;
        return;
    }
    // ids in order: (CTA, thread, register)
    const int per_thread = (n + CL * T - 1) / (CL * T);
    const int beg = min((rank * T + tid) * per_thread, n);
    const int n_mine = min(per_thread, n - beg);
    uint32_t round = 0;

    float w[REGS];
    float m = -INFINITY;
#pragma unroll
    for (int j = 0; j < REGS; j++) {
        w[j] = j < n_mine ? z[beg + j] : -INFINITY;
        m = fmaxf(m, w[j]);
    }
    m = combine1<CL, T, true>(m, &sh, round);
    float part = 0.f;
#pragma unroll
    for (int j = 0; j < REGS; j++) {
        w[j] = j < n_mine ? expf((w[j] - m) * a.inv_temperature) : 0.f;
        part += w[j];
    }
    const float total = combine1<CL, T, false>(part, &sh, round);

    // the nucleus: everything above t and the first k ids at t
    float above_t, at_t;
    const uint32_t t_bits = threshold_search<CL, T>(sp_tab, w, per_thread, a.top_p * total, false, false, above_t, at_t, &sh, round);
    const float t = __uint_as_float(t_bits);
    const int n_eq_t = (int)(t > 0.f ? at_t / t + 0.5f : 0.f);
    int k = n_eq_t;
    if (t > 0.f) {
        k = (int)ceilf((a.top_p * total - above_t) / t);
        k = max(1, min(k, max(n_eq_t, 1)));
    }
    const float kept = t > 0.f ? above_t + (float)k * t : above_t;

    // the draw
    const float u = fminf(fmaxf(a.uniforms[b], 0.f), 0.99999994f);
    const float ts = u * kept;
    float above_v, at_v;
    const uint32_t v_bits = threshold_search<CL, T>(sp_tab, w, per_thread, ts, true, true, above_v, at_v, &sh, round);
    const float v = __uint_as_float(v_bits);
    int q = v > 0.f ? (int)floorf((ts - above_v) / v) : 0;
    q = max(q, 0);
    if (v_bits == t_bits) q = min(q, k - 1);

    // the q-th id (in id order) whose weight is v
    int cnt = 0;
#pragma unroll
    for (int j = 0; j < REGS; j++) cnt += (j < n_mine && __float_as_uint(w[j]) == v_bits) ? 1 : 0;
    const int lane = tid & 31, warp = tid >> 5;
    int incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) sh.i[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        const int s = lane < T / 32 ? sh.i[lane] : 0;
        int si = s;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, si, o);
            if (lane >= o) si += y;
        }
        sh.i[lane] = si - s;  // exclusive offset of each warp inside the CTA
        if (lane == 31) sh.cnt_part = si;
    }
    if (CL > 1) cg::this_cluster().sync();
    else __syncthreads();
    if (tid == 0) {
        int before_cta = 0, all = 0;
        for (int r = 0; r < CL; r++) {
            const int c = CL > 1 ? *cg::this_cluster().map_shared_rank(&sh.cnt_part, r) : sh.cnt_part;
            if (r < rank) before_cta += c;
            all += c;
        }
        sh.before_cta = before_cta;
        sh.all_eq = all;
    }
    __syncthreads();
    q = min(q, max(sh.all_eq - 1, 0));
    const int before = sh.before_cta + sh.i[warp] + incl - cnt;
    if (cnt > 0 && q >= before && q < before + cnt) {
        int seen = before, id = beg;
#pragma unroll
        for (int j = 0; j < REGS; j++)
            if (j < n_mine && __float_as_uint(w[j]) == v_bits) {
                if (seen == q) id = beg + j;
                seen++;
            }
        const int token = lo + id;
        if (a.token_out) a.token_out[b] = token;
        if (a.key_out) a.key_out[b] = argmax_key(0.f, token);
    }
    if (CL > 1) cg::this_cluster().sync();  // no CTA leaves while another may still read its shared memory
}

// One launch: a row per CTA or cluster of CTAs, T threads of REGS weights each.
template <int CL, int T, int REGS>
static cudaError_t launch_nucleus_form(const SampleArgs &a, int n, cudaStream_t st, bool pdl)
{
    static PerDevice<bool> ready_dev;
    bool &ready = ready_dev.here();
    const int smem = 16 * T * (int)sizeof(float);  // the per-thread bucket table
    if (!ready) {
        const cudaError_t e =
            cudaFuncSetAttribute(nucleus_sample_kernel<CL, T, REGS>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
        ready = true;
    }
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof cfg);
    cfg.gridDim = dim3(n * CL);
    cfg.blockDim = dim3(T);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    int na = 0;
    if (CL > 1) {
        attr[na].id = cudaLaunchAttributeClusterDimension;
        attr[na].val.clusterDim.x = CL;
        attr[na].val.clusterDim.y = 1;
        attr[na].val.clusterDim.z = 1;
        na++;
    }
    if (pdl) {
        attr[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[na].val.programmaticStreamSerializationAllowed = 1;
        na++;
    }
    cfg.attrs = attr;
    cfg.numAttrs = na;
    return cudaLaunchKernelEx(&cfg, nucleus_sample_kernel<CL, T, REGS>, a);
}

// Launches for n rows, one per modality; `has_text` / `has_speech` say which occur among the rows.
inline cudaError_t launch_nucleus_sample(SampleArgs a, int n, bool has_text, bool has_speech, cudaStream_t st, bool pdl,
                                         int64_t *n_launches)
{
    for (int mod = 0; mod < 2; mod++) {
        if (!(mod ? has_speech : has_text)) continue;
        const int range = mod ? a.Vs : a.Vt;
        a.only_modality = mod;
        const cudaError_t e =
            range <= SP_THREADS * SP_SHORT_REGS ? launch_nucleus_form<1, SP_THREADS, SP_SHORT_REGS>(a, n, st, pdl)
            : range <= SP_CTA_RANGE             ? launch_nucleus_form<1, SP_THREADS, SP_REGS>(a, n, st, pdl)
                                                : launch_nucleus_form<SP_CLUSTER, SP_THREADS, SP_REGS>(a, n, st, pdl);
        if (e != cudaSuccess) return e;
        if (n_launches) (*n_launches)++;
    }
    return cudaSuccess;
}

}  // namespace sparsk
