// Attention phase of the persistent layer-range kernel and the merge of its partials (see sparsk_mega.cuh).
#pragma once

namespace sparsk {

// A warp's view of a run's ring items: items sub, sub + nsub, ... of the run, two 16-position tiles each (K and
// V, with the 128-byte swizzle, as the producers' TMA copies leave them), in the form attn_item_t asks for.
// The tiles were on their way before this launch's q/k/v projection had written the current rows' keys and
// values: those rows are copied over from the cache, and value rows past the end are cleared (they meet a
// weight of exactly zero, which must not meet a NaN).  Every warp that reads a tile does both for itself.
template <int HD, int SLOTS>
struct MkTiles {
    static constexpr int TILE = AT_TP * HD;   // numbers of one matrix's tile
    unsigned char *ring;
    MkShared *sh;
    int *status;
    const kv_t *kbase, *vbase;    // the cache of (slot, kv head)
    MkPos<SLOTS> at0;             // ring place of the run's first tiles
    int tile0, sub, nsub;
    int new0, end;                // the pass's own positions: [new0, end), end = the prefix's length
    int arrivals;                 // this warp's share of a slot's release
    int w_end;                    // no position from here on counts
    int n_tiles, lane;

    __device__ __forceinline__ static int off(int row, int c) { return at_swz<HD>(row, c); }
    __device__ __forceinline__ int item(int t) const { return sub + nsub * (t >> 1); }
    __device__ __forceinline__ MkPos<SLOTS> place(int t) const
    {
        MkPos<SLOTS> p = at0;
        p.skip_many(item(t));
        return p;
    }
    __device__ __forceinline__ int pos(int t) const { return (tile0 + 2 * item(t) + (t & 1)) * AT_TP; }
    __device__ __forceinline__ bool wait(int t, const kv_t *&Kt, const kv_t *&Vt) const
    {
        const MkPos<SLOTS> at = place(t);
        if (!(t & 1) && !mbar_wait(&sh->full[at.s], at.ph, &sh->giving_up, status)) return false;
        kv_t *kt = reinterpret_cast<kv_t *>(ring + (size_t)at.s * MK_SLOT_BYTES) + (t & 1) * 2 * TILE, *vt = kt + TILE;
        const int p0 = pos(t);
        if (p0 + AT_TP > new0) {
            constexpr int CH = HD / 8;
            for (int k = lane; k < AT_TP * CH; k += 32) {
                const int r = k / CH, c = k % CH, p = p0 + r;
                if (p < new0) continue;
                const size_t o = (size_t)p * HD + c * 8;
                if (p < end) *reinterpret_cast<uint4 *>(&kt[off(r, c)]) = __ldcg(reinterpret_cast<const uint4 *>(kbase + o));
                *reinterpret_cast<uint4 *>(&vt[off(r, c)]) = p < end ? __ldcg(reinterpret_cast<const uint4 *>(vbase + o)) : make_uint4(0u, 0u, 0u, 0u);
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
// Where it leaves its partial: the run's place in global memory, or the area, when several warps share the run.
template <int HD>
struct MkCells {
    float *po;
    float2 *pml;
    __device__ __forceinline__ float *o(int qg) const { return po + (ptrdiff_t)qg * HD; }
    __device__ __forceinline__ float2 *ml(int qg) const { return pml + qg; }
};
// One warp's partial of a block of eight query vectors and its sums.
template <int HD>
__host__ __device__ constexpr int mk_cell_bytes() { return 8 * HD * 4 + 8 * 8; }
// Shapes the phase can run: a warp per block of query vectors of a group.
inline bool mk_attn_fits(int M, int G) { return (M * G + 7) / 8 <= MK_CW; }

// The CTA's runs, one after another.  Up to four warps per block of eight query vectors share a run (as many as the area
// has room for partials, and two slots at least each), every nsub-th slot each; their partials meet in the area.
// (Blocks of sixteen, positions as columns, cost 450 bytes of spills, and a reload behind a grid barrier is a trip to the L2: flushes of
// four rows of the 28-layer shape 96.6 us a layer, so 90.9.)  Short runs go side by side, a warp per block.
template <int M, int HD, bool WIDE, int SLOTS>
__device__ __forceinline__ void mk_attention(const MkArgs &a, int l, unsigned char *area, unsigned char *ring, MkShared *sh,
                                             MkPos<SLOTS> &at)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, G = a.Hq / a.Hkv;
    AttnArgs aa{};
    aa.q32 = a.q_buf; aa.Hq = a.Hq; aa.Hkv = a.Hkv;
    const int stride = mk_part_rows(a), end = sh->att_t1;
    int t = sh->att_t0;
    MkRun r = sh->runs[0];
    const int batch = M == 1 ? 0 : sh->att_batch; // (one row has one group: its runs are long or alone)
    while (t < end) {
        int n_items = (r.n + 1) / 2, nsub = 1, sub = 0, qb = warp, before = 0;  // items before this warp's run
        if (M > 1 && batch > 1) {
            // (no more slots than the ring has, so none of them is filled twice before the warps meet again)
            static_assert(2 * MK_RUNS <= SLOTS, "slots of a batch");
            int mine = -1, w0 = 0;
            n_items = 0;
            for (int i = 0; i < batch; i++) {
                const int nb = sh->runs[i].n_qblk;
                if (warp >= w0 && warp < w0 + nb) {
                    mine = i;
                    qb = warp - w0;
                    before = n_items;
                }
                w0 += nb;
                n_items += (sh->runs[i].n + 1) / 2;
            }
            if (mine >= 0) r = sh->runs[mine];
            else sub = 1;
        } else {
            nsub = min(4, (n_items + 1) / 2);
            if (nsub > 1) {
                const int room = mk_area_bytes(M, WIDE) / (r.n_qblk * mk_cell_bytes<HD>());
                nsub = max(1, min(nsub, min(MK_CW / r.n_qblk, room)));
            }
            if (SLOTS % nsub) nsub = 2;  // a slot's successive fills stay with one warp
            if (r.n_qblk > 1) {
                sub = warp / r.n_qblk;
                qb = warp - sub * r.n_qblk;
            } else {
                sub = warp;
                qb = 0;
            }
        }
        const int nq = r.nq, n_qblk = r.n_qblk, run_items = (r.n + 1) / 2;
        const size_t part = (size_t)(blockIdx.x + r.g * a.Hkv + r.hk) * stride;
        if (sub < nsub) {
            AtItem item;
            item.qb = qb; item.hk = r.hk; item.row0 = r.row0; item.nrows = r.nrows; item.pos0 = r.pos0; item.nq = nq;
            const int w_end = min(r.pos0 + (r.nrows == 1 ? 0 : (min(qb * 8 + 8, nq) - 1) / G) + 1, a.S);
            MkTiles<HD, SLOTS> tiles;
            tiles.ring = ring; tiles.sh = sh; tiles.status = a.status;
            tiles.kbase = a.kc + l * a.kv_layer + (size_t)r.cache0 * HD; tiles.vbase = a.vc + l * a.kv_layer + (size_t)r.cache0 * HD;
            tiles.at0 = at;
            tiles.at0.skip_many(before);
            tiles.tile0 = r.tile0; tiles.sub = sub; tiles.nsub = nsub;
            tiles.new0 = r.pos0; tiles.end = min(r.pos0 + r.nrows, a.S);
            tiles.arrivals = qb == 0 ? MK_CW - (n_qblk - 1) : 1;
            const int mine = nsub == 1 ? run_items : (run_items - sub + nsub - 1) / nsub;
            tiles.n_tiles = 2 * mine - ((r.n & 1) && sub + nsub * (mine - 1) == run_items - 1 ? 1 : 0);
            tiles.lane = lane; tiles.w_end = w_end;
            MkCells<HD> out;
            if (nsub > 1) {
                // query vector qg of block qb at row qg - 8 qb of the warp's cells
                unsigned char *c = area + (size_t)(sub * n_qblk + qb) * mk_cell_bytes<HD>();
                out.po = reinterpret_cast<float *>(c) - (ptrdiff_t)qb * 8 * HD;
                out.pml = reinterpret_cast<float2 *>(c + 8 * HD * 4) - qb * 8;
            } else {
                out.po = a.part_o + part * HD;
                out.pml = a.part_ml + part;
            }
            attn_item_t<HD>(aa, item, nullptr, lane, nullptr, &tiles, &out);
        }
        at.skip_many(n_items);
        mk_consumer_sync();
        if (nsub > 1) {
            for (int k = threadIdx.x; k < nq * (HD / 4); k += MK_CW * 32) {
                const int qg = k / (HD / 4), c4 = k % (HD / 4), blk = qg / 8, ql = qg % 8;
                float mx = -INFINITY, sum = 0.f;
                float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
                for (int s = 0; s < nsub; s++)
                    mx = fmaxf(mx, reinterpret_cast<const float2 *>(area + (size_t)(s * n_qblk + blk) * mk_cell_bytes<HD>() + 8 * HD * 4)[ql].x);
                for (int s = 0; s < nsub; s++) {
                    const unsigned char *c = area + (size_t)(s * n_qblk + blk) * mk_cell_bytes<HD>();
                    const float2 ml = reinterpret_cast<const float2 *>(c + 8 * HD * 4)[ql];
                    const float w = ml.x == -INFINITY ? 0.f : __expf(ml.x - mx);
                    const float4 p = reinterpret_cast<const float4 *>(c)[ql * (HD / 4) + c4];
                    sum += ml.y * w;
                    o.x += p.x * w; o.y += p.y * w; o.z += p.z * w; o.w += p.w * w;
                }
                *reinterpret_cast<float4 *>(a.part_o + (part + qg) * HD + c4 * 4) = o;
                if (c4 == 0) a.part_ml[part + qg] = make_float2(mx, sum);
            }
            mk_consumer_sync();  // the next run may use the area
        }
        if (batch > 1) break;
        t += r.n;
        if (t < end) mk_run_at(a, sh, t, end, r);
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
