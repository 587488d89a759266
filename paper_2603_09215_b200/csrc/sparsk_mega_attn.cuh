// Attention phase of the persistent layer-range kernel and the merge of its partials (see sparsk_mega.cuh).
#pragma once

namespace sparsk {

// A warp's view of a run's ring items: items first, first + nsub, ... behind `at`, two 16-position tiles each (K and
// V, with the 128-byte swizzle, as the producers' TMA copies leave them), in the form attn_item_t asks for.
// The tiles were on their way before this launch's q/k/v projection had written the current rows' keys and
// values: those rows are copied over from the cache, and value rows past the end are cleared (they meet a
// weight of exactly zero, which must not meet a NaN).  Every warp that reads a tile does both for itself.
// What only a run's last tile or its end asks for is read from the run then: registers held across the tiles are spilled elsewhere, and a
// reload behind a grid barrier is a trip to the L2.
template <int HD, int SLOTS>
struct MkTiles {
    static constexpr int TILE = AT_TP * HD;   // numbers of one matrix's tile
    const MkArgs &a;
    const MkRun *r;
    MkShared *sh;
    unsigned char *ring;
    const MkPos<SLOTS> &at;       // the ring's place of item 0
    int layer, lane;
    int first, nsub;
    int tile0;                    // first tile of item 0
    int new0, w_end;              // the pass's own positions begin; no position from here on counts
    int arrivals;                 // this warp's share of a slot's release
    int n_tiles;

    __device__ __forceinline__ static int off(int row, int c) { return at_swz<HD>(row, c); }
    __device__ __forceinline__ int item(int t) const { return first + nsub * (t >> 1); }
    __device__ __forceinline__ MkPos<SLOTS> place(int t) const
    {
        MkPos<SLOTS> p = at;
        p.skip_many(item(t));
        return p;
    }
    __device__ __forceinline__ int pos(int t) const { return (tile0 + 2 * item(t) + (t & 1)) * AT_TP; }
    __device__ __forceinline__ bool wait(int t, const kv_t *&Kt, const kv_t *&Vt) const
    {
        const MkPos<SLOTS> p = place(t);
        if (!(t & 1) && !mbar_wait(&sh->full[p.s], p.ph, &sh->giving_up, a.status)) return false;
        kv_t *kt = reinterpret_cast<kv_t *>(ring + (size_t)p.s * MK_SLOT_BYTES) + (t & 1) * 2 * TILE, *vt = kt + TILE;
        const int p0 = pos(t);
        if (p0 + AT_TP > new0) {
            constexpr int CH = HD / 8;
            const int end = min(new0 + r->nrows, a.S);
            const size_t base = layer * a.kv_layer + (size_t)r->cache0 * HD;
            for (int k = lane; k < AT_TP * CH; k += 32) {
                const int row = k / CH, c = k % CH, q = p0 + row;
                if (q < new0) continue;
                const size_t o = base + (size_t)q * HD + c * 8;
                if (q < end) *reinterpret_cast<uint4 *>(&kt[off(row, c)]) = __ldcg(reinterpret_cast<const uint4 *>(a.kc + o));
                *reinterpret_cast<uint4 *>(&vt[off(row, c)]) = q < end ? __ldcg(reinterpret_cast<const uint4 *>(a.vc + o)) : make_uint4(0u, 0u, 0u, 0u);
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // before the slot's next copy
        }
        __syncwarp();
        Kt = kt;
        Vt = vt;
        return true;
    }
    __device__ __forceinline__ void release(int t) const
    {
        __syncwarp();
        if ((t & 1) || t == n_tiles - 1) {
            if (lane == 0) mbar_arrive_n(&sh->empty[place(t).s], (uint32_t)arrivals);
        }
    }
    __device__ __forceinline__ void start() const {}
    __device__ __forceinline__ void finish() const {}
};
// Where it leaves its partial: the run's place in global memory, or, when several warps share the run, the warp's cell in the area.
template <int HD>
struct MkCells {
    const MkArgs &a;
    const MkRun *r;
    unsigned char *cell;
    __device__ __forceinline__ float *o(int qg) const
    {
        return r->nsub > 1 ? reinterpret_cast<float *>(cell) + (qg % 8) * HD : a.part_o + (size_t)(r->part + qg) * HD;
    }
    __device__ __forceinline__ float2 *ml(int qg) const
    {
        return r->nsub > 1 ? reinterpret_cast<float2 *>(cell + 8 * HD * 4) + qg % 8 : a.part_ml + r->part + qg;
    }
};
// One warp's partial of a block of eight query vectors and its sums.
template <int HD>
__host__ __device__ constexpr int mk_cell_bytes() { return 8 * HD * 4 + 8 * 8; }

// The run that begins with tile t of the CTA's share, on its own: up to four warps per block of eight query vectors share it (as many as the
// area has room for partials, and two slots at least each), every nsub-th slot each.
template <int M, int HD, bool WIDE>
__device__ __forceinline__ void mk_run_alone(const MkArgs &a, MkShared *sh, int t, MkRun &r)
{
    constexpr int WARPS = mk_area_bytes(M, WIDE) / mk_cell_bytes<HD>() < MK_CW ? mk_area_bytes(M, WIDE) / mk_cell_bytes<HD>() : MK_CW;
    mk_run_at(a, sh, t, sh->att_t1, r);
    r.t = t;
    r.warp0 = r.item0 = 0;
    r.part = (int)(blockIdx.x + r.g * a.Hkv + r.hk) * mk_part_rows(a);
    r.nsub = max(1, min(min(4, ((r.n + 1) / 2 + 1) / 2), WARPS / r.n_qblk));
    if (mk_slots(M, WIDE) % r.nsub) r.nsub = 2;  // a slot's successive fills stay with one warp
}
// The first runs of the CTA (lane 0 of one warp, once a launch).  Are they worked on side by side?  If there are several, the ring holds all their
// tiles (so none of its slots is filled twice before the warps meet again), and a warp per block of query vectors is to be had: then
// with as many warps a block as above, or half as many, as long as there are warps and room for their partials.
template <int M, int HD, bool WIDE>
__device__ __forceinline__ void mk_runs(const MkArgs &a, MkShared *sh)
{
    constexpr int ROOM = mk_area_bytes(M, WIDE) / mk_cell_bytes<HD>();
    int t = sh->att_t0, n = 0, items = 0, blocks = 0;
    for (; n < MK_RUNS && t < sh->att_t1; n++) {
        MkRun &r = sh->runs[n];
        mk_run_alone<M, HD, WIDE>(a, sh, t, r);
        t += r.n;
        items += (r.n + 1) / 2;
        blocks += r.n_qblk;
    }
    sh->att_batch = t >= sh->att_t1 && n > 1 && items <= mk_slots(M, WIDE) && blocks <= MK_CW ? n : 0;
    if (!sh->att_batch) return;
    for (int want = 4, warps = MK_CW + 1; want >= 1 && warps > min(MK_CW, ROOM); want /= 2) {
        warps = items = 0;
        for (int i = 0; i < n; i++) {
            MkRun &r = sh->runs[i];
            r.nsub = min(want, ((r.n + 1) / 2 + 1) / 2);
            r.warp0 = warps;
            r.item0 = items;
            warps += r.nsub * r.n_qblk;
            items += (r.n + 1) / 2;
        }
    }
}

// The n query vectors of a run whose `nb` blocks of eight had `nsub` warps each: their partials, merged, to number `part`.
template <int HD>
__device__ __forceinline__ void mk_meet(const MkArgs &a, const unsigned char *cells, int nb, int nsub, int n, size_t part)
{
    for (int k = threadIdx.x; k < n * (HD / 4); k += MK_CW * 32) {
        const int ql = k / (HD / 4), c4 = k % (HD / 4);
        const unsigned char *first = cells + (size_t)(ql / 8) * mk_cell_bytes<HD>();
        float mx = -INFINITY, sum = 0.f;
        float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int s = 0; s < nsub; s++)
            mx = fmaxf(mx, reinterpret_cast<const float2 *>(first + (size_t)s * nb * mk_cell_bytes<HD>() + 8 * HD * 4)[ql % 8].x);
        for (int s = 0; s < nsub; s++) {
            const unsigned char *c = first + (size_t)s * nb * mk_cell_bytes<HD>();
            const float2 ml = reinterpret_cast<const float2 *>(c + 8 * HD * 4)[ql % 8];
            const float w = ml.x == -INFINITY ? 0.f : __expf(ml.x - mx);
            const float4 p = reinterpret_cast<const float4 *>(c)[ql % 8 * (HD / 4) + c4];
            sum += ml.y * w;
            o.x += p.x * w; o.y += p.y * w; o.z += p.z * w; o.w += p.w * w;
        }
        *reinterpret_cast<float4 *>(a.part_o + (part + ql) * HD + c4 * 4) = o;
        if (c4 == 0) a.part_ml[part + ql] = make_float2(mx, sum);
    }
}

// The CTA's runs: side by side, or one after another (mk_runs); the partials of warps that share a run meet in the area.  More
// than sixteen blocks have the run come by once for every sixteen.
// (Blocks of sixteen, positions as columns, cost 450 bytes of spills, and a reload behind a grid barrier is a trip to the L2: flushes of
// four rows of the 28-layer shape 96.6 us a layer, so 90.9.)
template <int M, int HD, bool WIDE, int SLOTS>
__device__ __forceinline__ void mk_attention(const MkArgs &a, int l, unsigned char *area, unsigned char *ring, MkShared *sh,
                                             MkPos<SLOTS> &at)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, G = a.Hq / a.Hkv;
    AttnArgs aa{};
    aa.q32 = a.q_buf; aa.Hq = a.Hq; aa.Hkv = a.Hkv;
    if (sh->att_t0 >= sh->att_t1) return;
    // Nothing of a run is held in registers across its tiles: it is read from shared memory before and after.  The one behind it is
    // worked out beside it, in the last three places in turn (whoever is late may still read the one before).
    static_assert(MK_RUNS == 4, "places");
    for (int at_run = 0, qb0 = 0;;) {  // qb0: first block of query vectors
        {
            const MkRun *r = &sh->runs[at_run];
            if (const int batch = sh->att_batch) {
                for (int i = 1; i < batch; i++)
                    if (warp >= sh->runs[i].warp0) r = &sh->runs[i];
            } else if (threadIdx.x == (MK_CW - 1) * 32 && r->t + r->n < sh->att_t1) {
                mk_run_alone<M, HD, WIDE>(a, sh, r->t + r->n, sh->runs[at_run == 3 ? 1 : at_run + 1]);
            }
            const int nb = min(MK_CW, r->n_qblk - qb0), nsub = r->nsub, in_run = warp - r->warp0, sub = nb > 1 ? in_run / nb : in_run;
            if (sub < nsub) {
                const int qb = qb0 + (nb > 1 ? in_run - sub * nb : 0);
                AtItem item;
                item.qb = qb; item.hk = r->hk; item.row0 = r->row0; item.nrows = r->nrows; item.pos0 = r->pos0; item.nq = r->nq;
                MkTiles<HD, SLOTS> tiles{a, r, sh, ring, at, l, lane};
                tiles.first = r->item0 + sub; tiles.nsub = nsub; tiles.tile0 = r->tile0 - 2 * r->item0;
                tiles.new0 = r->pos0;
                tiles.w_end = min(r->pos0 + (r->nrows == 1 ? 0 : (min(qb * 8 + 8, r->nq) - 1) / G) + 1, a.S);
                tiles.arrivals = qb == qb0 ? MK_CW - (nb - 1) : 1;
                const int run_items = (r->n + 1) / 2, mine = nsub == 1 ? run_items : (run_items - sub + nsub - 1) / nsub;
                tiles.n_tiles = 2 * mine - ((r->n & 1) && sub + nsub * (mine - 1) == run_items - 1 ? 1 : 0);
                const MkCells<HD> out{a, r, area + (size_t)warp * mk_cell_bytes<HD>()};
                attn_item_t<HD>(aa, item, nullptr, lane, nullptr, &tiles, &out);
            }
        }
        mk_consumer_sync();
        const int batch = sh->att_batch;
        const MkRun *r = &sh->runs[batch ? batch - 1 : at_run];  // (the last of several)
        at.skip_many(r->item0 + (r->n + 1) / 2);
        bool met = false;
        for (int i = batch ? 0 : at_run; i <= (batch ? batch - 1 : at_run); i++) {
            const MkRun *b = &sh->runs[i];
            if (b->nsub > 1) {
                mk_meet<HD>(a, area + (size_t)b->warp0 * mk_cell_bytes<HD>(), b->n_qblk, b->nsub, b->nq, (size_t)b->part);
                met = true;
            }
        }
        if (batch) break;
        if ((qb0 += MK_CW) >= r->n_qblk) {
            if (r->t + r->n >= sh->att_t1) break;
            qb0 = 0;
            at_run = at_run == 3 ? 1 : at_run + 1;
        }
        if (met) mk_consumer_sync();  // what comes next may use the area
    }
}

__device__ __forceinline__ MkMerge mk_merge_of(const MkArgs &a, const MkShared *sh, int h, int m)
{
    MkMerge r{0, -1, 0};
    const int G = a.Hq / a.Hkv, hk = h / G;
    const int g = m < a.n_rows && h < a.Hq ? sh->row_grp[m] : -1, tiles = g >= 0 ? sh->grp_tiles[g] : 0;
    if (tiles > 0) {
        const int t0 = sh->att_base[g] + hk * tiles;
        r.cf = mk_run_cta(sh, t0);
        r.cl = mk_run_cta(sh, t0 + tiles - 1);
        r.cell0 = (g * a.Hkv + hk) * mk_part_rows(a) + (m - sh->grp_row0[g]) * G + h - hk * G;
    }
    return r;
}
// Merge of the partials of query heads hq and, with NH = 2, hq + 1, for all rows: 16 / (M NH) warps per row and head, a
// share of the partials each, then the shares meet in scr.  Leaves the output of head i, row m at column c
// through put(i, m, c, value).
template <int M, int HD, int NH, class Put>
__device__ __forceinline__ void mk_merge_heads(const MkArgs &a, const MkShared *sh, int hq, float *scr, const Put &put)
{
    constexpr int WPR = MK_CW / (M * NH), LN = HD / 4;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int hm = warp / WPR, m = hm % M, wi = warp % WPR, stride = mk_part_rows(a);
    float2 *scr_ml = reinterpret_cast<float2 *>(scr + MK_CW * HD);
    float mx = -INFINITY, l = 0.f;
    float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
    const MkMerge p = hq == sh->head0 ? sh->merge[hm / M][m] : mk_merge_of(a, sh, hq + hm / M, m);
    {
        const int cl = p.cl;
        constexpr int U = 5;
        for (int c0 = p.cf + wi; c0 <= cl; c0 += WPR * U) {
            float2 ml[U];
            float4 v[U];
#pragma unroll
            for (int u = 0; u < U; u++) {
                const int c = c0 + u * WPR;
                const size_t cell = (size_t)(p.cell0 + c * stride);
                ml[u] = c <= cl ? a.part_ml[cell] : make_float2(-INFINITY, 0.f);
                v[u] = c <= cl && lane < LN ? reinterpret_cast<const float4 *>(a.part_o + cell * HD)[lane] : make_float4(0.f, 0.f, 0.f, 0.f);
            }
            float top = mx;
#pragma unroll
            for (int u = 0; u < U; u++) top = fmaxf(top, ml[u].x);
            if (top == -INFINITY) continue;  // (the same in all lanes)
            const float old = __expf(mx - top);
            l *= old;
            o.x *= old; o.y *= old; o.z *= old; o.w *= old;
#pragma unroll
            for (int u = 0; u < U; u++) {
                const float w = ml[u].x == -INFINITY ? 0.f : __expf(ml[u].x - top);
                l += ml[u].y * w;
                o.x += v[u].x * w; o.y += v[u].y * w; o.z += v[u].z * w; o.w += v[u].w * w;
            }
            mx = top;
        }
    }
    if (lane < LN) reinterpret_cast<float4 *>(scr + warp * HD)[lane] = o;
    if (lane == 0) scr_ml[warp] = make_float2(mx, l);
    mk_consumer_sync();
    for (int k = threadIdx.x; k < NH * M * HD; k += MK_CW * 32) {
        const int at = k / HD, c = k % HD;
        float top = -INFINITY, den = 0.f, num = 0.f;
#pragma unroll
        for (int w = 0; w < WPR; w++) top = fmaxf(top, scr_ml[at * WPR + w].x);
#pragma unroll
        for (int w = 0; w < WPR; w++) {
            const float2 ml = scr_ml[at * WPR + w];
            const float f = ml.x == -INFINITY ? 0.f : __expf(ml.x - top);
            den += ml.y * f;
            num += scr[(at * WPR + w) * HD + c] * f;
        }
        put(at / M, at % M, c, den > 0.f ? num / den : 0.f);
    }
    mk_consumer_sync();
}

}  // namespace sparsk
