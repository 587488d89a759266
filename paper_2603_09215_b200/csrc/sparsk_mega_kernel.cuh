// The persistent layer-range kernel itself (see sparsk_mega.cuh).
#pragma once

namespace sparsk {

// ------------------------------------------------------------------ producers
// One producer warp: walks the CTA's ring items in consumption order and issues every fourth.
template <int M, int HD, bool WIDE>
__device__ __forceinline__ void mk_produce(const MkArgs &a, unsigned char *ring, MkShared *sh, int p)
{
    constexpr int SLOTS = mk_slots(M, WIDE);
    constexpr bool TC = M >= MK_TC_ROWS;
    const int lane = threadIdx.x & 31;
    uint32_t idx = 0;   // ring item
    bool ok = true;
    // waits until item idx's slot is free and no more than `flight` items (counting this one) are on
    // their way, and announces `bytes`; item idx - flight was this warp's own
    const uint32_t few = M == 1 && !WIDE && sh->bands[0].end <= (int)gridDim.x ? MK_FEW_IN_FLIGHT : MK_IN_FLIGHT;
    uint32_t flight = few;
    static_assert(MK_IN_FLIGHT % MK_PW == 0 && MK_FEW_IN_FLIGHT % MK_PW == 0 && SLOTS % MK_PW == 0, "a producer waits for items of its own");
    auto open = [&](uint32_t bytes) {
        const int s = idx % SLOTS;
        int go = 1;
        if (lane == 0) {
            if (SLOTS > (int)flight && idx >= flight) {
                const uint32_t o = idx - flight;
                go = mbar_wait(&sh->full[o % SLOTS], (o / SLOTS) & 1, &sh->giving_up, a.status) ? 1 : 0;
            }
            if (go) go = mbar_wait(&sh->empty[s], ((idx / SLOTS) & 1) ^ 1, &sh->giving_up, a.status) ? 1 : 0;
            if (go) mbar_expect_tx(&sh->full[s], bytes);
        }
        ok = __shfl_sync(0xffffffffu, go, 0) != 0;
        return ok;
    };
    auto rows = [&](int type, const MkLayer *L) {
        MkBands w = sh->bands[type == MK_QKV ? 0 : 1];
        const uint32_t idx0 = idx, bytes = MK_SLOT_BYTES + (type == MK_QKV && L - a.layers == a.short_copy_layer && blockIdx.x == 0 ? 16 : 0);
        flight = few;
        for (; w.j < w.end; w.j += w.step)
            for (int ks = 0; ks < w.k_steps; ks++, idx++) {
                if (idx - idx0 == SLOTS && type == MK_MLP) flight = MK_IN_FLIGHT;
                if ((int)(idx % MK_PW) != p) continue;
                if (!open(bytes)) return;
                if (lane < 2) {
                    const CUtensorMap *map;
                    int row;
                    mk_band(type, a, L, w.j, lane, map, row);
                    const int s = idx % SLOTS;
                    const uint32_t dst = smem_u32(ring) + s * MK_SLOT_BYTES + lane * MK_BOX_BYTES;
                    // (three and four rows: the same box as four swizzled 64-column blocks)
                    if (TC) tma_load_3d(dst, map + MKW_N, &sh->full[s], 0, row, ks * (MK_BOX_COLS / 64));
                    else tma_load_2d(dst, map, &sh->full[s], ks * MK_BOX_COLS, row);
                }
            }
    };
    auto column_box = [&](const CUtensorMap *map, int cols, int col0, int row0) {
        if ((int)(idx % MK_PW) == p) {
            if (!open((uint32_t)(MK_CBOX_ROWS * cols * 2))) return;
            if (lane == 0) {
                const int s = idx % SLOTS;
                const uint32_t dst = smem_u32(ring) + s * MK_SLOT_BYTES;
                if (TC) tma_load_3d(dst, map + MKW_N, &sh->full[s], 0, row0, col0 / 32);
                else tma_load_2d(dst, map, &sh->full[s], col0, row0);
            }
        }
        idx++;
    };
    for (int l = a.layer_begin; l < a.layer_end && ok; l++) {
        const MkLayer *L = a.layers + l;
        rows(MK_QKV, L);
        if (!ok) break;
        MkRun r = sh->runs[0];
        for (int t = sh->att_t0, qb0 = 0; ok && t < sh->att_t1;) {
            if (t != sh->att_t0 && qb0 == 0) mk_run_at(a, sh, t, sh->att_t1, r);
            if ((qb0 += MK_CW) >= r.n_qblk) {  // (as often as it takes to have every block of query vectors see it)
                t += r.n;
                qb0 = 0;
            }
            const int y0 = r.cache0;
            for (int i = 0; i < r.n; i += 2, idx++) {
                if ((int)(idx % MK_PW) != p) continue;
                const int n = min(2, r.n - i);
                if (!open((uint32_t)(n * 2 * AT_TP * HD * sizeof(kv_t)))) break;
                if (lane < 2 * n) {
                    const int s = idx % SLOTS, y = y0 + (r.tile0 + i + (lane >> 1)) * AT_TP;
                    const uint32_t dst = smem_u32(ring) + s * MK_SLOT_BYTES + lane * (AT_TP * HD * (uint32_t)sizeof(kv_t));
                    const CUtensorMap *map = lane & 1 ? &L->vmap : &L->kmap;
                    if (HD > 64) tma_load_3d(dst, map, &sh->full[s], 0, y, 0);
                    else tma_load_2d(dst, map, &sh->full[s], 0, y);
                }
            }
        }
        if (!ok) break;
        const MkPairs w = sh->heads;
        for (int i = w.lo; i < w.hi && ok; i++) column_box(&L->map[MKW_O], HD, (i / w.boxes) * HD, (i % w.boxes) * MK_CBOX_ROWS);
        if (!ok) break;
        rows(MK_MLP, L);
        if (!ok) break;
        if constexpr (WIDE) {
            const MkPairs v = sh->downs;
            for (int i = v.lo; i < v.hi && ok; i++) column_box(&L->map[MKW_D], MK_CBOX_COLS, (i / v.boxes) * MK_CBOX_COLS, (i % v.boxes) * MK_CBOX_ROWS);
        } else {
            const MkBands b = sh->bands[1];
            if (b.j < b.end)
                for (int i = 0; i < w.boxes && ok; i++) column_box(&L->map[MKW_D], a.cols.box, b.j * MK_BOX_ROWS, i * MK_CBOX_ROWS);
        }
    }
    // never leave with copies in flight: every slot this producer filled must have landed
    // (consumers that gave up no longer free slots, so wait on the full barriers, 2 ms each)
    if (lane == 0) {
        const uint32_t total = idx;  // items before the point where this producer stopped
        for (int s = p; s < SLOTS; s += MK_PW)
            if (total > (uint32_t)s) mbar_wait(&sh->full[s], ((total - 1 - s) / SLOTS) & 1, &sh->never, nullptr, 2000000ull);
    }
}

// ------------------------------------------------------------------ consumers: O-projection and MLP
template <int M, int HD, int SLOTS>
__device__ __forceinline__ void mk_oproj(const MkArgs &a, unsigned char *area, unsigned char *ring, MkShared *sh, MkPos<SLOTS> &at)
{
    const MkPairs w = sh->heads;
    constexpr bool TC = M >= MK_TC_ROWS;
    constexpr int RS = HD + 8;
    // two merged heads, as fp32 rows or as two planes each
    float *const x = reinterpret_cast<float *>(area);
    bf16 *const planes = reinterpret_cast<bf16 *>(area);
    float *scr = reinterpret_cast<float *>(area + 8 * 1024);
    static_assert((TC ? 2 * 2 * M * RS * 2 : 2 * M * HD * 4) <= 8 * 1024, "two heads' activations");
    auto put = [&](int i, int m, int c, float v) {
        if constexpr (TC) mk_put_planes<M>(planes + i * 2 * M * RS, RS, m, c, v);
        else x[(i * M + m) * HD + c] = v;
    };
    // a share reaches into a second head as often as not, into a third one only with more heads than CTAs
    for (int i = w.lo; i < w.hi;) {
        const int hq = i == w.lo ? sh->head0 : i / w.boxes;
        if (i != w.lo) mk_consumer_sync();  // everyone is done with the heads before
        if ((hq + 1) * w.boxes < w.hi) mk_merge_heads<M, HD, 2>(a, sh, hq, scr, put);
        else mk_merge_heads<M, HD, 1>(a, sh, hq, scr, put);
        for (int k = 0; k < 2 && i < w.hi; k++) {
            const int r0 = i - (hq + k) * w.boxes, n = min(w.boxes - r0, w.hi - i);
            if constexpr (TC) mk_columns_tc<M>(a, a.h, r0, r0 + n, HD, planes + k * 2 * M * RS, RS, ring, sh, at);
            else mk_columns<M, HD / 8>(a, a.h, r0, r0 + n, HD, x + k * M * HD, HD, ring, sh, at);
            i += n;
            at.skip_many(n);
        }
    }
}

// Gate/up, and in the narrow form the down-projection of what the CTA's own bands made.
template <int M, bool WIDE, int SLOTS>
__device__ __forceinline__ void mk_mlp(const MkArgs &a, int l, const bf16 *gain, unsigned char *area, unsigned char *ring, MkShared *sh,
                                       const MkGains &gains, MkPos<SLOTS> &at)
{
    const int boxes = (a.d + MK_CBOX_ROWS - 1) / MK_CBOX_ROWS;
    const MkBands w = sh->bands[1];
    if (w.j >= w.end) return;
    // columns of the box that are the next CTA's meet zeros
    if constexpr (M >= MK_TC_ROWS) {
        constexpr int RS = MK_CBOX_COLS + 8;
        bf16 *planes = reinterpret_cast<bf16 *>(area);
        float *red = reinterpret_cast<float *>(area + mk_tc_planes_bytes(M, w.k_steps * MK_BOX_COLS));
        bf16 *u = reinterpret_cast<bf16 *>(reinterpret_cast<unsigned char *>(red) + MK_TC_RED_BYTES);
        if (!WIDE)
            for (int i = threadIdx.x; i < M * RS; i += MK_CW * 32) reinterpret_cast<uint32_t *>(u)[i] = 0u;
        mk_rows_tc<M, WIDE>(MK_MLP, a, l, planes, red, nullptr, gain, gains, u, RS, ring, sh, at);
        if constexpr (!WIDE) {
            mk_consumer_sync();
            mk_columns_tc<M>(a, a.h2, 0, boxes, a.cols.box, u, RS, ring, sh, at);
            at.skip_many(boxes);
        }
    } else if constexpr (WIDE) {
        mk_rows<M, true>(MK_MLP, a, l, reinterpret_cast<float *>(area), reinterpret_cast<float *>(area + mk_area_bytes(M, true) - mk_sums_bytes(M)),
                         mk_act_window(M, true, mk_sums_bytes(M)), nullptr, gain, gains, nullptr, 0, ring, sh, at);
    } else {
        constexpr int OWN = M * MK_CBOX_COLS * 4 + mk_sums_bytes(M);
        static_assert(mk_act_window(M, false, OWN) >= MK_NARROW_STEPS, "the narrow form's rows are whole");
        float *u = reinterpret_cast<float *>(area + mk_area_bytes(M, false) - OWN), *sums = u + M * MK_CBOX_COLS;
        for (int i = threadIdx.x; i < M * MK_CBOX_COLS; i += MK_CW * 32) u[i] = 0.f;
        mk_rows<M, false>(MK_MLP, a, l, reinterpret_cast<float *>(area), sums, mk_act_window(M, false, OWN), nullptr, gain, gains, u, MK_CBOX_COLS, ring, sh, at);
        mk_consumer_sync();
        if (a.cols.box <= 64) mk_columns<M, 8>(a, a.h2, 0, boxes, a.cols.box, u, MK_CBOX_COLS, ring, sh, at);
        else mk_columns<M, 16>(a, a.h2, 0, boxes, a.cols.box, u, MK_CBOX_COLS, ring, sh, at);
        at.skip_many(boxes);
    }
}

// Wide form: the CTA's share of the down-projection, the activations of its blocks of 128 columns a few at a time.
template <int M, int SLOTS>
__device__ __forceinline__ void mk_down(const MkArgs &a, unsigned char *area, unsigned char *ring, MkShared *sh, MkPos<SLOTS> &at)
{
    constexpr bool TC = M >= MK_TC_ROWS;
    constexpr int C = MK_CBOX_COLS, RS = C + 8, NB = 4;
    const MkPairs w = sh->downs;
    float *const x = reinterpret_cast<float *>(area);
    bf16 *const planes = reinterpret_cast<bf16 *>(area);
    for (int i = w.lo; i < w.hi;) {
        const int b0 = i / w.boxes, nb = min(NB, (w.hi - 1) / w.boxes - b0 + 1);
        if (i != w.lo) mk_consumer_sync();  // everyone is done with the blocks before
        for (int k = threadIdx.x; k < nb * M * (C / 4); k += MK_CW * 32) {
            const int c = k % (C / 4) * 4, m = k / (C / 4) % M, b = k / (C / 4) / M, col = (b0 + b) * C + c;
            const float4 v = col < a.F && m < a.n_rows ? *reinterpret_cast<const float4 *>(a.act + (size_t)m * a.F + col) : make_float4(0.f, 0.f, 0.f, 0.f);
            if constexpr (TC) {
                uint2 hi, lo;
                split_pair(v.x, v.y, hi.x, lo.x);
                split_pair(v.z, v.w, hi.y, lo.y);
                *reinterpret_cast<uint2 *>(planes + (size_t)(b * 2 * M + m) * RS + c) = hi;
                *reinterpret_cast<uint2 *>(planes + (size_t)(b * 2 * M + M + m) * RS + c) = lo;
            } else {
                *reinterpret_cast<float4 *>(x + (b * M + m) * C + c) = v;
            }
        }
        mk_consumer_sync();
        for (int k = 0; k < nb; k++) {
            const int r0 = i - (b0 + k) * w.boxes, n = min(w.boxes - r0, w.hi - i);
            if constexpr (TC) mk_columns_tc<M>(a, a.h, r0, r0 + n, C, planes + k * 2 * M * RS, RS, ring, sh, at);
            else mk_columns<M, 16>(a, a.h, r0, r0 + n, C, x + k * M * C, C, ring, sh, at);
            i += n;
            at.skip_many(n);
        }
    }
}

// h += h2, h2 = 0: `n` threads of every CTA, this one the i-th of them.
__device__ __forceinline__ void mk_fold(const MkArgs &a, int i, int n)
{
    const int total = a.n_rows * a.d / 4;
    for (int k = (int)blockIdx.x + i * (int)gridDim.x; k < total; k += n * (int)gridDim.x) {
        float4 *p = reinterpret_cast<float4 *>(a.h) + k, *q = reinterpret_cast<float4 *>(a.h2) + k;
        const float4 x = *p, y = *q;
        *p = make_float4(x.x + y.x, x.y + y.y, x.z + y.z, x.w + y.w);
        *q = make_float4(0.f, 0.f, 0.f, 0.f);
    }
}

template <int M, int HD, bool WIDE>
__global__ void __launch_bounds__(MK_THREADS, 1) mega_kernel(const MkArgs a)
{
    constexpr int SLOTS = mk_slots(M, WIDE), AREA = mk_area_bytes(M, WIDE);
    extern __shared__ __align__(1024) unsigned char mk_smem[];  // (nothing else is in shared memory: the swizzled boxes need 1024)
    unsigned char *ring = mk_smem;
    unsigned char *area = ring + (size_t)SLOTS * MK_SLOT_BYTES;
    MkShared *sh = reinterpret_cast<MkShared *>(area + AREA);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < SLOTS; s++) {
            mbar_init(&sh->full[s], 1);
            mbar_init(&sh->empty[s], MK_CW);
        }
        sh->giving_up = 0;
        sh->never = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        if (lane < MK_MAX_ROWS) {
            const int i = lane;
            sh->row_slot[i] = i < a.n_rows ? a.row_slot[i] : -1;
            sh->row_pos[i] = i < a.n_rows ? a.row_pos[i] : -1;
            sh->row_grp[i] = -1;
            sh->grp_row0[i] = i < a.n_groups ? a.grp_row0[i] : -1;
            sh->grp_nrows[i] = i < a.n_groups ? a.grp_nrows[i] : 0;
        }
        __syncwarp();
        if (lane == 0) {
            int base = 0;
            for (int g = 0; g < MK_MAX_ROWS; g++) {
                const int r0 = sh->grp_row0[g], n = sh->grp_nrows[g];
                const bool sane = r0 >= 0 && n >= 1 && r0 + n <= a.n_rows && sh->row_slot[r0] >= 0 && sh->row_slot[r0] < a.n_slots &&
                                  sh->row_pos[r0] >= 0;
                const int tiles = sane ? (min(sh->row_pos[r0] + n, a.S) + AT_TP - 1) / AT_TP : 0;
                sh->grp_tiles[g] = tiles;
                sh->att_base[g] = base;
                base += tiles * a.Hkv;
                for (int r = 0; sane && r < n; r++) sh->row_grp[r0 + r] = g;
            }
            sh->att_base[MK_MAX_ROWS] = base;
            const unsigned n = (unsigned)min((int)gridDim.x, base), c = blockIdx.x;
            sh->att_ctas = (int)n;
            sh->att_t0 = c < n ? (int)(c * (unsigned)base / n) : 0;
            sh->att_t1 = c < n ? (int)((c + 1) * (unsigned)base / n) : 0;
            mk_runs<M, HD, WIDE>(a, sh);
            sh->bands[0].init(MK_QKV, a);
            sh->bands[1].init(MK_MLP, a);
            sh->heads.init(a, a.Hq);
            if (WIDE) sh->downs.init(a, (a.F + MK_CBOX_COLS - 1) / MK_CBOX_COLS);
            sh->head0 = sh->heads.lo / sh->heads.boxes;
        }
    }
    __syncthreads();
    if ((int)threadIdx.x < MK_BOX_ROWS * M)
        sh->fin[threadIdx.x] = mk_fin(a, sh, blockIdx.x, (int)threadIdx.x / M, (int)threadIdx.x % M);
    if (warp == MK_CW - 1 && lane < 2 * MK_MAX_ROWS)
        sh->merge[lane / MK_MAX_ROWS][lane % MK_MAX_ROWS] = mk_merge_of(a, sh, sh->head0 + lane / MK_MAX_ROWS, lane % MK_MAX_ROWS);
    __syncthreads();

    if (warp >= MK_CW) {
        mk_produce<M, HD, WIDE>(a, ring, sh, warp - MK_CW);
    } else {
        constexpr bool TC = M >= MK_TC_ROWS;
        MkPos<SLOTS> at{0, 0u};
        unsigned long long epoch = a.bar_base;
        if (blockIdx.x == 0 && threadIdx.x == 0 && a.trace) a.trace[0] = global_ns();
        bool ok = true;
        MkGains gains;
        const bf16 *gain = a.layers[a.layer_begin].attn_gain;
        gains.load(gain, a.d);
        for (int l = a.layer_begin; l < a.layer_end && ok; l++) {
            const bf16 *mlp_gain = a.layers[l].mlp_gain;
            const float *h2 = WIDE ? nullptr : a.h2;
            if constexpr (TC) {
                const int whole = (a.d + MK_BOX_COLS - 1) / MK_BOX_COLS * MK_BOX_COLS;
                mk_rows_tc<M, WIDE>(MK_QKV, a, l, reinterpret_cast<bf16 *>(area), reinterpret_cast<float *>(area + mk_tc_planes_bytes(M, whole)),
                                    h2, gain, gains, nullptr, 0, ring, sh, at);
            } else {
                mk_rows<M, WIDE>(MK_QKV, a, l, reinterpret_cast<float *>(area), reinterpret_cast<float *>(area + AREA - mk_sums_bytes(M)),
                                 mk_act_window(M, WIDE, mk_sums_bytes(M)), h2, gain, gains, nullptr, 0, ring, sh, at);
            }
            if (!(ok = mk_grid_barrier(a, sh, epoch))) break;
            if (!WIDE && warp == MK_CW - 1) mk_fold(a, lane, 32);
            mk_attention<M, HD, WIDE>(a, l, area, ring, sh, at);
            if (!(ok = mk_grid_barrier(a, sh, epoch))) break;
            mk_oproj<M, HD>(a, area, ring, sh, at);
            if (!(ok = mk_grid_barrier(a, sh, epoch, &gains, mlp_gain))) break;
            mk_mlp<M, WIDE>(a, l, mlp_gain, area, ring, sh, gains, at);
            if constexpr (WIDE) {
                if (!(ok = mk_grid_barrier(a, sh, epoch))) break;
                mk_down<M>(a, area, ring, sh, at);
            }
            gain = a.layers[min(l + 1, a.layer_end - 1)].attn_gain;
            ok = mk_grid_barrier(a, sh, epoch, &gains, gain);
        }
        if (ok && !WIDE) mk_fold(a, (int)threadIdx.x, MK_CW * 32);
    }
    __syncthreads();
}

}  // namespace sparsk
