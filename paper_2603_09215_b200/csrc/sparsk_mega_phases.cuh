// Projection phases of the persistent layer-range kernel (see sparsk_mega.cuh).
#pragma once

namespace sparsk {

// ------------------------------------------------------------------ activations -> shared memory
// Where column i (a multiple of 4) of a row sits inside the activation area.  A lane of a
// consumer warp needs the eight columns 8 lane .. 8 lane + 7 of a 256-column step (the columns of
// its 16-byte weight unit); read as two float4 at a 32-byte stride they would collide two ways on
// the banks, so each 256-column step is stored as two planes of 128 floats: columns 8 l + 0..3 at
// [4 l], columns 8 l + 4..7 at [128 + 4 l], and the two reads of a warp are both conflict-free.
__device__ __forceinline__ int mk_act_slot(int i)
{
    const int ci = i & (MK_BOX_COLS - 1);
    return (i - ci) + ((ci >> 2) & 1) * (MK_BOX_COLS / 2) + (ci >> 3) * 4;
}

// Four numbers of the residual stream from element i on: h, or h + h2 where the down-projection's sums have
// not been folded into h yet.
__device__ __forceinline__ float4 mk_resid(const float *h, const float *h2, size_t i)
{
    float4 v = *reinterpret_cast<const float4 *>(h + i);
    if (h2) {
        const float4 w = *reinterpret_cast<const float4 *>(h2 + i);
        v = make_float4(v.x + w.x, v.y + w.y, v.z + w.z, v.w + w.w);
    }
    return v;
}

// The gains a thread needs for the columns it keeps in registers in mk_norm.  They are cold (every layer's are read once a
// launch), so they are asked for while the CTA waits for the grid barrier before the norm.
constexpr int MK_KEEP = 2;
struct MkGains {
    uint2 g[MK_KEEP];
    __device__ __forceinline__ void load(const bf16 *gain, int K)
    {
#pragma unroll
        for (int k = 0; k < MK_KEEP; k++) {
            const int i = ((int)threadIdx.x + k * MK_CW * 32) * 4;
            g[k] = i < K ? *reinterpret_cast<const uint2 *>(gain + i) : make_uint2(0u, 0u);
        }
    }
};

// Consumers only: wait until every CTA has arrived at this barrier.  A warp whose wait for a ring slot ran out
// stays until here, without working, because the barriers among the CTA's warps have no time limit;
// here all of them learn of it and leave together.  The gains of the norm behind the barrier are asked for between
// arriving and waiting: a release waits for loads on their way as well.
__device__ __forceinline__ bool mk_grid_barrier(const MkArgs &a, MkShared *sh, unsigned long long &epoch, MkGains *gains = nullptr,
                                                const bf16 *gain = nullptr)
{
    mk_consumer_sync();
    epoch += gridDim.x;
    if (threadIdx.x == 0) {
        // release: everything this CTA wrote (ordered before by the CTA barrier) is visible to
        // whoever acquires the counter; no value comes back, so nothing waits on the round trip
        asm volatile("red.release.gpu.global.add.u64 [%0], %1;" ::"l"(a.bar), "l"(1ull) : "memory");
    }
    if (gains) gains->load(gain, a.d);
    if (threadIdx.x == 0) {
        unsigned long long t0 = 0;
        bool leave = false;
        for (uint32_t spin = 0;; ++spin) {
            if (ld_acquire_u64(a.bar) >= epoch) break;
            if ((spin & 63u) == 63u) {
                // this CTA or another (or an earlier launch that was never cleaned up after) gave up
                if ((leave = ld_volatile_i32(a.abort_word) || *(volatile int *)&sh->giving_up)) break;
                const unsigned long long now = global_ns();
                if (t0 == 0) t0 = now;
                else if ((leave = now - t0 > GM_TIMEOUT_NS)) break;
            }
        }
        if (leave || *(volatile int *)&sh->giving_up) {
            // say so, also where all have arrived (with a wait for a ring slot that ran out on the way here): skipping the rest
            // is never silent, and nobody sits out a time limit of his own at the next barrier
            sh->giving_up = 1;
            atomicOr(a.status, ST_TIMEOUT);
            atomicExch(a.abort_word, 1);
            leave = true;
        }
        sh->go_on = !leave;
        if (blockIdx.x == 0 && a.trace) a.trace[(epoch - a.bar_base) / gridDim.x] = global_ns();
    }
    mk_consumer_sync();
    return sh->go_on != 0;  // one answer for all warps
}

// x = (h + h2) / sqrt(mean((h + h2)^2) + eps) * gain for the M rows, left through put(row, column, four numbers); columns at
// or beyond K, up to ncols, and rows from n_rows on are zeros.  Rows of up to MK_KEEP float4s per thread stay in
// registers between the sum of squares and the scaling: one trip to the L2.  (Wider rows parked in the area
// meanwhile, instead of read again: no difference, 130 us a layer at one row of 5,120 numbers, 194 at 7,168.)
template <int M, class Put>
__device__ __forceinline__ void mk_norm(int ncols, int K, int n_rows, const float *h, const float *h2, const bf16 *gain,
                                        const MkGains &gains, float eps, MkShared *sh, const Put &put)
{
    constexpr int T = MK_CW * 32, KEEP = MK_KEEP;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    float4 v[M][KEEP];
    float ss[M];
#pragma unroll
    for (int k = 0; k < KEEP; k++)
#pragma unroll
        for (int m = 0; m < M; m++) {
            const int i = (tid + k * T) * 4;
            v[m][k] = i < K && m < n_rows ? mk_resid(h, h2, (size_t)m * K + i) : zero;
        }
#pragma unroll
    for (int m = 0; m < M; m++) {
        ss[m] = 0.f;
#pragma unroll
        for (int k = 0; k < KEEP; k++) ss[m] += v[m][k].x * v[m][k].x + v[m][k].y * v[m][k].y + v[m][k].z * v[m][k].z + v[m][k].w * v[m][k].w;
    }
    for (int i = (tid + KEEP * T) * 4; i < K; i += T * 4)
#pragma unroll
        for (int m = 0; m < M; m++) {
            if (m >= n_rows) break;
            const float4 x = mk_resid(h, h2, (size_t)m * K + i);
            ss[m] += x.x * x.x + x.y * x.y + x.z * x.z + x.w * x.w;
        }
#pragma unroll
    for (int m = 0; m < M; m++) {
        ss[m] = warp_sum(ss[m]);
        if (lane == 0) sh->red_rows[m][warp] = ss[m];
    }
    mk_consumer_sync();  // also: everyone is done with what the area held
    float inv[M];
#pragma unroll
    for (int m = 0; m < M; m++) {
        float tot = 0.f;
#pragma unroll
        for (int w = 0; w < MK_CW; w++) tot += sh->red_rows[m][w];
        inv[m] = rsqrtf(tot / (float)K + eps);
    }
    auto scaled = [&](int m, const float4 &x, const uint2 &g) {
        return make_float4(x.x * inv[m] * bf_lo(g.x), x.y * inv[m] * bf_hi(g.x), x.z * inv[m] * bf_lo(g.y), x.w * inv[m] * bf_hi(g.y));
    };
#pragma unroll
    for (int k = 0; k < KEEP; k++) {
        const int i = (tid + k * T) * 4;
        if (i >= ncols) continue;
#pragma unroll
        for (int m = 0; m < M; m++) put(m, i, scaled(m, v[m][k], gains.g[k]));
    }
    for (int i = (tid + KEEP * T) * 4; i < ncols; i += T * 4) {
        const uint2 g = i < K ? *reinterpret_cast<const uint2 *>(gain + i) : make_uint2(0u, 0u);
#pragma unroll
        for (int m = 0; m < M; m++) put(m, i, scaled(m, i < K && m < n_rows ? mk_resid(h, h2, (size_t)m * K + i) : zero, g));
    }
    mk_consumer_sync();
}

// Columns [c0, c0 + ncols) of M rows that do not fit the area whole, as fp32, row m at act + m * ncols (in the
// layout of mk_act_slot); ncols is a multiple of 256.
template <int M>
__device__ __forceinline__ void mk_norm_window(float *act, int c0, int ncols, int K, const float *h, const float *h2,
                                               const bf16 *gain, float eps, MkShared *sh)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int T = MK_CW * 32;
#pragma unroll
    for (int m = 0; m < M; m++) {
        const size_t row = (size_t)m * K;
        float ss = 0.f;
        for (int i = tid * 4; i < K; i += T * 4) {
            const float4 v = mk_resid(h, h2, row + i);
            ss += v.x * v.x + v.y * v.y + v.z * v.z + v.w * v.w;
        }
        ss = warp_sum(ss);
        if (lane == 0) sh->red_rows[m][warp] = ss;
    }
    mk_consumer_sync();  // also: everyone is done with what the area held
#pragma unroll
    for (int m = 0; m < M; m++) {
        const size_t row = (size_t)m * K;
        float *dst = act + (size_t)m * ncols;
        float tot = 0.f;
#pragma unroll
        for (int w = 0; w < MK_CW; w++) tot += sh->red_rows[m][w];
        const float inv = rsqrtf(tot / (float)K + eps);
        for (int i = tid * 4; i < ncols; i += T * 4) {
            float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
            const int k = c0 + i;
            if (k < K) {
                const float4 p = mk_resid(h, h2, row + k);
                const uint2 g2 = *reinterpret_cast<const uint2 *>(gain + k);
                o = make_float4(p.x * inv * bf_lo(g2.x), p.y * inv * bf_hi(g2.x), p.z * inv * bf_lo(g2.y),
                                p.w * inv * bf_hi(g2.y));
            }
            *reinterpret_cast<float4 *>(dst + mk_act_slot(i)) = o;
        }
    }
    mk_consumer_sync();
}

// Two fp32 numbers in a register pair; a * b + c on both at once.
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 mk_pair(float lo, float hi)
{
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ f32x2 mk_fma2(f32x2 a, f32x2 b, f32x2 c)
{
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ float mk_sum2(f32x2 a)
{
    float lo, hi;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(a));
    return lo + hi;
}
// eight bf16 weights as four pairs
__device__ __forceinline__ void mk_unpack(const uint4 &w, f32x2 (&p)[4])
{
    p[0] = mk_pair(bf_lo(w.x), bf_hi(w.x));
    p[1] = mk_pair(bf_lo(w.y), bf_hi(w.y));
    p[2] = mk_pair(bf_lo(w.z), bf_hi(w.z));
    p[3] = mk_pair(bf_lo(w.w), bf_hi(w.w));
}

// The sums over LANES neighbouring lanes of N <= LANES numbers each (powers of two).  After every step a lane holds
// half as many sums, each of twice as many lanes; in the end sum k is v[0] of the LANES / N lanes from LANES / N * k on.
template <int N, int LANES>
__device__ __forceinline__ void mk_exchange(float (&v)[N], int lane)
{
    int off = LANES / 2;
#pragma unroll
    for (int n = N / 2; n > 0; n >>= 1, off >>= 1) {
        const bool up = lane & off;
#pragma unroll
        for (int k = 0; k < N / 2; k++) {
            if (k >= n) break;
            const float give = up ? v[k] : v[k + n], keep = up ? v[k + n] : v[k];
            v[k] = keep + __shfl_xor_sync(0xffffffffu, give, off);
        }
    }
#pragma unroll
    for (; off > 0; off >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], off);
}

// ------------------------------------------------------------------ what a finished pair of sums becomes
// Row `rib` of the two boxes of q/k/v band b, for activation row m.
__device__ __forceinline__ MkFin mk_fin(const MkArgs &a, const MkShared *sh, int b, int rib, int m)
{
    MkFin f{make_float2(1.f, 0.f), 0, 0, MK_FIN_NONE};
    if (m >= a.n_rows) return f;
    const int half = a.hd >> 1, per_head = half / MK_BOX_ROWS;
    const int nq = a.Hq * per_head, nk = a.Hkv * per_head;
    const int pos = sh->row_pos[m];
    const size_t row = (size_t)sh->row_slot[m] * a.Hkv;
    if (b < nq + nk) {
        const int bb = b < nq ? b : b - nq;
        const int head = bb / per_head, i = (bb % per_head) * MK_BOX_ROWS + rib;
        f.cs = a.rope[(size_t)pos * half + i];
        f.second = half;
        f.kind = b < nq ? MK_FIN_Q : MK_FIN_K;
        f.off = b < nq ? ((size_t)m * a.Hq + head) * a.hd + i : ((row + head) * a.S + pos) * a.hd + i;
    } else {
        const int n = (b - nq - nk) * 2 * MK_BOX_ROWS + rib;   // (a head is a multiple of 32 numbers: n + 16 is in the same)
        f.second = MK_BOX_ROWS;
        f.kind = n < a.Hkv * a.hd ? MK_FIN_V : MK_FIN_NONE;
        f.off = ((row + n / a.hd) * a.S + pos) * a.hd + n % a.hd;
    }
    return f;
}
__device__ __forceinline__ void mk_finish_qkv(const MkArgs &a, int l, const MkFin &f, float v0, float v1)
{
    const float ra = v0 * f.cs.x - v1 * f.cs.y, rb = v1 * f.cs.x + v0 * f.cs.y;
    if (f.kind == MK_FIN_Q) {
        a.q_buf[f.off] = ra;
        a.q_buf[f.off + f.second] = rb;
    } else if (f.kind == MK_FIN_K) {
        kv_t *dst = a.kc + l * a.kv_layer + f.off;
        dst[0] = to_kv(ra);
        dst[f.second] = to_kv(rb);
    } else if (f.kind == MK_FIN_V) {
        kv_t *dst = a.vc + l * a.kv_layer + f.off;
        dst[0] = to_kv(v0);
        dst[f.second] = to_kv(v1);
    }
}
__device__ __forceinline__ float mk_silu_mul(float gate, float up) { return gate / (1.f + __expf(-gate)) * up; }

// ------------------------------------------------------------------ one and two rows
// Waits for a slot and takes eight 16-byte units per lane out of it: `stride` bytes apart, the second four from `second` on.  The
// slot is free for its next fill before its products are formed.  False: the wait ran out.
template <int SLOTS>
__device__ __forceinline__ bool mk_take(uint4 (&w)[8], const unsigned char *ring, MkShared *sh, const MkPos<SLOTS> &p, int off, int stride,
                                        int second, int *status)
{
    if (!mbar_wait(&sh->full[p.s], p.ph, &sh->giving_up, status)) return false;
    const unsigned char *src = ring + (size_t)p.s * MK_SLOT_BYTES + off;
#pragma unroll
    for (int r = 0; r < 8; r++) w[r] = *reinterpret_cast<const uint4 *>(src + (r >= 4 ? second : 0) + (r & 3) * stride);
    __syncwarp();
    if ((threadIdx.x & 31) == 0) mbar_arrive_n(&sh->empty[p.s], MK_CW / MK_GROUPS);
    return true;
}

// Row form.  A slot s is the work of the four warps of group s mod 4, four rows of both boxes each; the groups' sums of a row
// meet in shared memory once per eight bands.  (All sixteen warps on every slot, a row of both boxes each, took
// 0.35 us a slot from a full ring, as long as HBM takes to fill it; in groups 0.2: a warp spends some ten cycles an
// instruction, and waiting, releasing and reading the activations cost as much as the products.)
// `room` k-steps of M rows fit the area.  If that is the whole inner dimension they are loaded once; otherwise (WIDE only) the area
// holds a window that is reloaded as the phase moves along.  gate/up leaves its results in u: column
// (band - first band) * 16 + row of the box, of activation row m at u + m * u_stride; WIDE: in a.act.
constexpr int MK_BATCH = 8;  // bands whose sums wait in shared memory
__host__ __device__ constexpr int mk_sums_bytes(int M) { return MK_BATCH * 2 * MK_BOX_ROWS * M * MK_GROUPS * 4; }

template <int M, bool WIDE, int SLOTS>
__device__ __forceinline__ void mk_rows(int type, const MkArgs &a, int l, float *act, float *sums, int room, const float *h2,
                                        const bf16 *gain, const MkGains &gains, float *u, int u_stride, unsigned char *ring,
                                        MkShared *sh, MkPos<SLOTS> &at)
{
    constexpr int ROWS = MK_BOX_ROWS / (MK_CW / MK_GROUPS), N = 2 * ROWS * M;  // rows of a box per warp; sums per warp
    static_assert(ROWS == 4, "mk_take");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, grp = warp / MK_GROUPS, sub = warp % MK_GROUPS;
    MkBands w = sh->bands[type == MK_QKV ? 0 : 1];
    if (w.j >= w.end) return;
    const int first = w.j, n_bands = (w.end - w.j + w.step - 1) / w.step;
    const bool whole = !WIDE || w.k_steps <= room;
    const int window = whole ? w.k_steps : room, ncols = window * MK_BOX_COLS;
    bool live = true;        // false: a wait ran out, this warp only keeps the barriers whole
    if (whole)
        mk_norm<M>(ncols, a.d, a.n_rows, a.h, h2, gain, gains, a.eps, sh,
                   [&](int m, int i, const float4 &x) { *reinterpret_cast<float4 *>(act + (size_t)m * ncols + mk_act_slot(i)) = x; });
    for (int b0 = 0; b0 < n_bands; b0 += MK_BATCH) {
        const int nb = min(MK_BATCH, n_bands - b0);
        for (int b = 0; b < nb; b++) {
            f32x2 acc[2 * ROWS][M];
#pragma unroll
            for (int r = 0; r < 2 * ROWS; r++)
#pragma unroll
                for (int m = 0; m < M; m++) acc[r][m] = 0ull;
            for (int win0 = 0; win0 < w.k_steps; win0 += window) {
                const int n = min(window, w.k_steps - win0);
                if (!whole) mk_norm_window<M>(act, win0 * MK_BOX_COLS, ncols, a.d, a.h, h2, gain, a.eps, sh);
                const int ahead = (grp - at.s) & (MK_GROUPS - 1);
                MkPos<SLOTS> p = at;
                p.skip(ahead);
                for (int k = ahead; k < n && live; k += MK_GROUPS, p.skip(MK_GROUPS)) {
                    uint4 wt[2 * ROWS];
                    if (!(live = mk_take(wt, ring, sh, p, sub * ROWS * MK_BOX_COLS * 2 + lane * 16, MK_BOX_COLS * 2, MK_BOX_BYTES, a.status))) break;
                    f32x2 xv[M][4];
#pragma unroll
                    for (int m = 0; m < M; m++) {
                        const float *xp = act + (size_t)m * ncols + k * MK_BOX_COLS + lane * 4;
                        const ulonglong2 xa = *reinterpret_cast<const ulonglong2 *>(xp), xb = *reinterpret_cast<const ulonglong2 *>(xp + MK_BOX_COLS / 2);
                        xv[m][0] = xa.x; xv[m][1] = xa.y; xv[m][2] = xb.x; xv[m][3] = xb.y;
                    }
#pragma unroll
                    for (int r = 0; r < 2 * ROWS; r++) {
                        f32x2 wp[4];
                        mk_unpack(wt[r], wp);
#pragma unroll
                        for (int m = 0; m < M; m++)
#pragma unroll
                            for (int j = 0; j < 4; j++) acc[r][m] = mk_fma2(wp[j], xv[m][j], acc[r][m]);
                    }
                }
                at.skip_many(n);
            }
            float v[N];
#pragma unroll
            for (int r = 0; r < 2 * ROWS; r++)
#pragma unroll
                for (int m = 0; m < M; m++) v[r * M + m] = mk_sum2(acc[r][m]);
            mk_exchange<N, 32>(v, lane);
            // sum k of N sits in the 32 / N lanes from 32 / N k on
            const int k = lane / (32 / N), r = k / M, m = k % M;
            if (lane % (32 / N) == 0)
                sums[((b * 2 * MK_BOX_ROWS + (r / ROWS) * MK_BOX_ROWS + sub * ROWS + r % ROWS) * M + m) * MK_GROUPS + grp] = v[0];
        }
        mk_consumer_sync();
        for (int i = threadIdx.x; i < nb * MK_BOX_ROWS * M; i += MK_CW * 32) {
            const int m = i % M, rib = i / M % MK_BOX_ROWS, b = i / M / MK_BOX_ROWS;
            const float4 s0 = reinterpret_cast<const float4 *>(sums)[(b * 2 * MK_BOX_ROWS + rib) * M + m];
            const float4 s1 = reinterpret_cast<const float4 *>(sums)[(b * 2 * MK_BOX_ROWS + MK_BOX_ROWS + rib) * M + m];
            const float v0 = (s0.x + s0.y) + (s0.z + s0.w), v1 = (s1.x + s1.y) + (s1.z + s1.w);
            if (type == MK_QKV) mk_finish_qkv(a, l, b0 + b == 0 ? sh->fin[i] : mk_fin(a, sh, first + (b0 + b) * w.step, rib, m), v0, v1);
            else if (!WIDE) u[m * u_stride + (b0 + b) * MK_BOX_ROWS + rib] = mk_silu_mul(v0, v1);
            else if (const int c = (first + (b0 + b) * w.step) * MK_BOX_ROWS + rib; c < a.F) a.act[(size_t)m * a.F + c] = mk_silu_mul(v0, v1);
        }
        if (b0 + MK_BATCH < n_bands) mk_consumer_sync();
    }
}

// Column form.
// Boxes [r0, r1) of 64 weight rows x `cols` columns, the first of them at ring place `at`: dst[m][row] += W[row][its
// columns] . x_m, x_m (cols numbers) at x + m * x_stride in shared memory.  A slot s is the work of the four
// warps of group s mod 4, sixteen rows each.  LPR lanes share a row, eight columns each, whose activations they hold
// in registers: the products of a box need nothing but the weights from shared memory, and the sums of
// sixteen rows meet in 8 (one row of activations) or 15 (two) shuffles.
template <int M, int LPR, int SLOTS>
__device__ __forceinline__ void mk_columns(const MkArgs &a, float *dst, int r0, int r1, int cols, const float *x, int x_stride,
                                           unsigned char *ring, MkShared *sh, MkPos<SLOTS> at)
{
    constexpr int RPL = 32 / LPR, NL = 16 / RPL;  // rows per load, loads per box
    static_assert(NL <= 8, "mk_take");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, grp = warp / MK_GROUPS, sub = warp % MK_GROUPS;
    const int li = lane & (LPR - 1), row_in = lane / LPR;
    const bool on = li * 8 < cols;
    f32x2 xv[M][4];
#pragma unroll
    for (int m = 0; m < M; m++) {
        const ulonglong2 z = make_ulonglong2(0ull, 0ull);
        const ulonglong2 xa = on ? *reinterpret_cast<const ulonglong2 *>(x + m * x_stride + li * 8) : z;
        const ulonglong2 xb = on ? *reinterpret_cast<const ulonglong2 *>(x + m * x_stride + li * 8 + 4) : z;
        xv[m][0] = xa.x; xv[m][1] = xa.y; xv[m][2] = xb.x; xv[m][3] = xb.y;
    }
    // (lanes without columns read their row's first ones, and drop them)
    const int ahead = (grp - at.s) & (MK_GROUPS - 1), stride = RPL * cols * 2, off = (sub * 16 + row_in) * cols * 2 + (on ? li * 16 : 0);
    at.skip(ahead);
    for (int r = r0 + ahead; r < r1; r += MK_GROUPS, at.skip(MK_GROUPS)) {
        uint4 wt[8];
        if (!mk_take(wt, ring, sh, at, off, stride, NL > 4 ? 4 * stride : 0, a.status)) return;
        float v[NL * M];
#pragma unroll
        for (int i = 0; i < NL; i++) {
            f32x2 w[4];
            mk_unpack(on ? wt[i] : make_uint4(0u, 0u, 0u, 0u), w);
#pragma unroll
            for (int m = 0; m < M; m++) {
                f32x2 t = mk_fma2(w[0], xv[m][0], 0ull);
#pragma unroll
                for (int j = 1; j < 4; j++) t = mk_fma2(w[j], xv[m][j], t);
                v[i * M + m] = mk_sum2(t);
            }
        }
        // NL * M = LPR / 2 * M sums over LPR lanes: one each with two activation rows, one per pair of lanes with one
        mk_exchange<NL * M, LPR>(v, lane);
        const int m = M == 1 ? 0 : li & 1, row = r * MK_CBOX_ROWS + sub * 16 + (li >> 1) * RPL + row_in;
        if ((M == 2 || !(li & 1)) && row < a.d) atomicAdd(dst + (size_t)m * a.d + row, v[0]);
    }
}

// ------------------------------------------------------------------ three and four rows: tensor-core form
// The same two forms with mma.sync m16n8k16: A = 16 weight rows x 16 columns (ldmatrix, conflict-free under the
// copies' swizzle), B = 16 columns x 8 columns of which the first M are the rows' hi terms and the next M their lo
// terms (two bf16 terms, 16 significant bits, as on the tcgen05 path): one instruction for both, added at
// the end.  In the row form a warp of a slot's four takes one box and half of its columns, and the eight shares of a
// box (four groups, two halves) meet in shared memory at the end of a band.
constexpr int MK_TC_RED_BYTES = 2 * 2 * 8 * 16 * 8 * 4;  // [parity][box][share][16 rows][8 n] floats = 16 KB
// The area with three and four rows: planes of d columns, the band sums, planes of the CTA's own columns.
__host__ __device__ constexpr size_t mk_tc_planes_bytes(int M, int cols) { return (size_t)2 * M * (cols + 8) * 2; }
constexpr int MK_TC_STEPS = 17;  // k-steps of a residual row
static_assert(mk_tc_planes_bytes(MK_MAX_ROWS, MK_TC_STEPS * MK_BOX_COLS) + MK_TC_RED_BYTES + mk_tc_planes_bytes(MK_MAX_ROWS, MK_CBOX_COLS) <=
                  (size_t)mk_area_bytes(MK_MAX_ROWS, false), "planes");
__device__ __forceinline__ void mma_bf16_16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// Column c of activation row m as two bf16 terms, in planes of M rows: hi rows, then lo rows.
template <int M>
__device__ __forceinline__ void mk_put_planes(bf16 *planes, int rs, int m, int c, float x)
{
    const bf16 hi = __float2bfloat16(x);
    planes[(size_t)m * rs + c] = hi;
    planes[(size_t)(M + m) * rs + c] = __float2bfloat16(x - __bfloat162float(hi));
}
__device__ __forceinline__ void ldsm_x4(uint32_t (&r)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr)
                 : "memory");
}

// Row form.  gate/up leaves its results as planes of their own, u_planes, row stride u_rs; WIDE: as fp32 in a.act.
template <int M, bool WIDE, int SLOTS>
__device__ __forceinline__ void mk_rows_tc(int type, const MkArgs &a, int l, bf16 *planes, float *red, const float *h2,
                                           const bf16 *gain, const MkGains &gains, bf16 *u_planes, int u_rs, unsigned char *ring,
                                           MkShared *sh, MkPos<SLOTS> &at)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int g = lane >> 2, t = lane & 3;
    const int grp = warp / MK_GROUPS, box = (warp >> 1) & 1, half = warp & 1;
    MkBands w = sh->bands[type == MK_QKV ? 0 : 1];
    if (w.j >= w.end) return;
    // row stride: the padding spreads the rows over the banks
    const int first = w.j, ncols = w.k_steps * MK_BOX_COLS, rs = ncols + 8;
    mk_norm<M>(ncols, a.d, a.n_rows, a.h, h2, gain, gains, a.eps, sh, [&](int m, int i, const float4 &x) {
        uint2 hi, lo;
        split_pair(x.x, x.y, hi.x, lo.x);
        split_pair(x.z, x.w, hi.y, lo.y);
        *reinterpret_cast<uint2 *>(planes + (size_t)m * rs + i) = hi;
        *reinterpret_cast<uint2 *>(planes + (size_t)(M + m) * rs + i) = lo;
    });
    // this lane's row address inside a 64-column block for ldmatrix: matrices (rows 0-7, k 0-7),
    // (rows 8-15, k 0-7), (rows 0-7, k 8-15), (rows 8-15, k 8-15)
    const int lrow = (lane & 7) + ((lane >> 3) & 1) * 8, lchk = lane >> 4;
    const uint32_t a_off = (uint32_t)box * MK_BOX_BYTES + (uint32_t)half * (2 * MK_BOX_ROWS * 128) + (uint32_t)lrow * 128;
    const bf16 *act = planes + (size_t)g * rs + half * 128 + 2 * t;
    static_assert(2 * M == 8, "a plane row per column of the B operand");
    uint32_t band_it = 0;
    bool live = true;        // false: a wait ran out, this warp only keeps the barriers whole
    for (; w.j < w.end; w.j += w.step) {
        float acc[4] = {0.f, 0.f, 0.f, 0.f}, acc2[4] = {0.f, 0.f, 0.f, 0.f};
        const int ahead = (grp - at.s) & (MK_GROUPS - 1);
        MkPos<SLOTS> p = at;
        p.skip(ahead);
        for (int ks = ahead; ks < w.k_steps && live; ks += MK_GROUPS, p.skip(MK_GROUPS)) {
            if (!(live = mbar_wait(&sh->full[p.s], p.ph, &sh->giving_up, a.status))) break;
            const uint32_t slot = smem_u32(ring) + (uint32_t)p.s * MK_SLOT_BYTES + a_off;
            const bf16 *bp = act + ks * MK_BOX_COLS;
            uint32_t af[8][4];
#pragma unroll
            for (int j = 0; j < 8; j++)
                ldsm_x4(af[j], slot + (uint32_t)(j >> 2) * (MK_BOX_ROWS * 128) + (((uint32_t)((j & 3) * 2 + lchk) ^ (uint32_t)(lrow & 7)) << 4));
            __syncwarp();
            if (lane == 0) mbar_arrive_n(&sh->empty[p.s], MK_CW / MK_GROUPS);
#pragma unroll
            for (int j = 0; j < 8; j++) {
                const uint32_t b0 = *reinterpret_cast<const uint32_t *>(bp + j * 16), b1 = *reinterpret_cast<const uint32_t *>(bp + j * 16 + 8);
                if (j & 1) mma_bf16_16816(acc2, af[j], b0, b1);
                else mma_bf16_16816(acc, af[j], b0, b1);
            }
        }
        at.skip_many(w.k_steps);
#pragma unroll
        for (int e = 0; e < 4; e++) acc[e] += acc2[e];
        // the eight shares of each box meet: [parity][box][share][16 rows][8 n]
        float *mine = red + ((((band_it & 1) * 2 + box) * 8 + grp * 2 + half) * 16) * 8;
        *reinterpret_cast<float2 *>(mine + g * 8 + 2 * t) = make_float2(acc[0], acc[1]);
        *reinterpret_cast<float2 *>(mine + (g + 8) * 8 + 2 * t) = make_float2(acc[2], acc[3]);
        mk_consumer_sync();
        if (threadIdx.x < MK_BOX_ROWS * M) {
            const int rib = threadIdx.x / M, m = threadIdx.x % M;
            const float *r0 = red + (((band_it & 1) * 2 + 0) * 8 * 16) * 8 + rib * 8 + m;
            const float *r1 = red + (((band_it & 1) * 2 + 1) * 8 * 16) * 8 + rib * 8 + m;
            float v0 = 0.f, v1 = 0.f;
#pragma unroll
            for (int sl = 0; sl < 8; sl++) {
                v0 += r0[sl * 16 * 8] + r0[sl * 16 * 8 + M];
                v1 += r1[sl * 16 * 8] + r1[sl * 16 * 8 + M];
            }
            if (type == MK_QKV) {
                mk_finish_qkv(a, l, band_it == 0 ? sh->fin[threadIdx.x] : mk_fin(a, sh, w.j, rib, m), v0, v1);
            } else if (WIDE) {
                if (const int c = w.j * MK_BOX_ROWS + rib; c < a.F) a.act[(size_t)m * a.F + c] = mk_silu_mul(v0, v1);
            } else {
                const int c = (w.j - first) * MK_BOX_ROWS + rib;
                mk_put_planes<M>(u_planes, u_rs, m, c, mk_silu_mul(v0, v1));  // (rows beyond n_rows: their planes are zeros)
            }
        }
        band_it++;
    }
}

// Column form (see mk_columns): a warp's sixteen rows are the A operand, the activations of the columns sit in
// registers as B operands, and a box's sums need no other warp.  x: planes of M rows, row stride x_rs.
template <int M, int SLOTS>
__device__ __forceinline__ void mk_columns_tc(const MkArgs &a, float *dst, int r0, int r1, int cols, const bf16 *x, int x_rs,
                                              unsigned char *ring, MkShared *sh, MkPos<SLOTS> at)
{
    constexpr int KS = MK_CBOX_COLS / 16;
    static_assert(2 * M == 8, "the exchange below adds column n + M to column n");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, grp = warp / MK_GROUPS, sub = warp % MK_GROUPS;
    const int g = lane >> 2, t = lane & 3, nk = cols / 16;
    uint32_t b[KS][2];
#pragma unroll
    for (int k = 0; k < KS; k++) {
        b[k][0] = b[k][1] = 0u;
        if (k < nk) {
            b[k][0] = *reinterpret_cast<const uint32_t *>(x + (size_t)g * x_rs + k * 16 + 2 * t);
            b[k][1] = *reinterpret_cast<const uint32_t *>(x + (size_t)g * x_rs + k * 16 + 8 + 2 * t);
        }
    }
    const int lrow = sub * 16 + (lane & 7) + ((lane >> 3) & 1) * 8, lchk = lane >> 4;
    const int ahead = (grp - at.s) & (MK_GROUPS - 1);
    at.skip(ahead);
    for (int r = r0 + ahead; r < r1; r += MK_GROUPS, at.skip(MK_GROUPS)) {
        if (!mbar_wait(&sh->full[at.s], at.ph, &sh->giving_up, a.status)) return;
        const uint32_t slot = smem_u32(ring) + (uint32_t)at.s * MK_SLOT_BYTES + (uint32_t)lrow * 64;
        float acc[4] = {0.f, 0.f, 0.f, 0.f}, acc2[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int k = 0; k < KS; k++) {
            if (k < nk) {
                uint32_t af[4];
                const uint32_t chunk = (uint32_t)((k & 1) * 2 + lchk);
                ldsm_x4(af, slot + (uint32_t)(k >> 1) * (MK_CBOX_ROWS * 64) + ((chunk ^ (uint32_t)((lrow >> 1) & 3)) << 4));
                if (k & 1) mma_bf16_16816(acc2, af, b[k][0], b[k][1]);
                else mma_bf16_16816(acc, af, b[k][0], b[k][1]);
            }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive_n(&sh->empty[at.s], MK_CW / MK_GROUPS);
        // lanes t < 2 hold hi terms of rows 2 t and 2 t + 1, lanes t + 2 the lo terms of the same; the lower ones finish weight row g,
        // the upper ones g + 8
#pragma unroll
        for (int e = 0; e < 4; e++) acc[e] += acc2[e];
        const bool up = t >= 2;
        const float y0 = (up ? acc[2] : acc[0]) + __shfl_xor_sync(0xffffffffu, up ? acc[0] : acc[2], 2);
        const float y1 = (up ? acc[3] : acc[1]) + __shfl_xor_sync(0xffffffffu, up ? acc[1] : acc[3], 2);
        const int row = r * MK_CBOX_ROWS + sub * 16 + g + (up ? 8 : 0), m = (t & 1) * 2;
        if (row < a.d) {
            if (m < a.n_rows) atomicAdd(dst + (size_t)m * a.d + row, y0);
            if (m + 1 < a.n_rows) atomicAdd(dst + (size_t)(m + 1) * a.d + row, y1);
        }
    }
}

}  // namespace sparsk

#include "sparsk_mega_attn.cuh"
#include "sparsk_mega_kernel.cuh"
