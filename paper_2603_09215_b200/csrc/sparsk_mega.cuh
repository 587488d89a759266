// Persistent layer-range kernel for passes of one to four rows.
//
// At so few rows a decode step is nothing but a stream of weights from HBM (Sec. IV-B.3),
// and one kernel per projection leaves HBM idle at every kernel boundary.  This kernel runs a
// whole range of layers in ONE cooperative launch, one CTA per SM:
//
//   * warps 16..19 are producers.  They walk the same list of work as everyone else but only
//     ever look at weights and at the cache, which depend on nothing this launch computes (the few
//     cache rows that do are patched in by their readers), so they keep TMA copies flowing into a
//     ring of 16 KB shared-memory slots across phase and layer boundaries.  Producer p owns the
//     slots p, p + 4, ... and cycles them on its own (one thread needs a few hundred nanoseconds
//     per copy, so four run side by side).  The ring is what keeps HBM streaming while the
//     consumers sit in a barrier.  Twelve slots cover 4.2 us of HBM; no more than eight are on
//     their way at once (148 SMs, 16 KB boxes from HBM: 6.1 / 6.9 / 7.03 / 6.6 TB/s with 4 / 6 / 8 / 12
//     slots on their way, 7.01 with twelve slots of which eight are).
//     (Asking the L2 for weights further ahead was measured in three forms and lost each time:
//     tensor or bulk prefetches running ahead of the copies made every phase slower, gate/up by
//     30-80 %; a burst for the next gate/up bands during the attention phases delayed the
//     attention's own cache reads by as much as it later saved.)
//   * warps 0..15 are consumers.  Per layer they run four phases separated by grid-wide barriers:
//     RMSNorm + q/k/v + rotary embedding + cache append; attention partials; O-projection;
//     RMSNorm + gate/up + SiLU + down-projection (a phase of its own in the wide form, see MkCols).
//     - Row form (q/k/v, gate/up: a sum is needed whole before anything can be done with it): a
//       CTA owns "bands" of 32 weight rows in two 16-row boxes (rotary pairs, gate/up pairs, or
//       plain rows) over the whole inner dimension.
//     - Column form (O, down: sums that are added to the residual stream): a CTA owns columns of the
//       matrix, i.e. a stretch of the inner dimension, for many or all weight rows, and adds its
//       share of every output.  So it needs only the few activations of its columns, which sit in
//       registers: of the attention output the one or two heads it owns, whose splits it merges for
//       itself (no merge phase), and of the MLP activation exactly what its own gate/up bands made
//       (no barrier between gate/up and down).  The additions of the 148 CTAs to one row are 0.6 us
//       of L2 atomics beside a stream of 20.
//     Activations are fp32 (three and four rows: two bf16 terms of 16 significant bits, see
//     sparsk_mega_phases.cuh): at random initialisation a rounding early in the stack is amplified by
//     every later layer, and bf16 activations alone put the exit states of a 28-layer stack 2-3 %
//     from the fp64 reference.
//     While some CTA still reads the residual stream at the start of the MLP, another may be done with
//     its gate/up bands: the down-projection therefore adds into a buffer of its own (h2), which the
//     next layer's first RMSNorm reads along with h and the attention phase folds into h.  (Not in the wide form.)
//
// Every wait (ring slot, grid barrier) is bounded by a wall-clock limit; on a timeout the CTA
// raises ST_TIMEOUT, tells the other CTAs through the abort word, lets its copies land and
// returns.
#pragma once

#include <cstddef>

#include "sparsk_attn.cuh"
#include "sparsk_gemm.cuh"

namespace sparsk {

constexpr int MK_CW = 16;                       // consumer warps
constexpr int MK_PW = 4;                        // producer warps
constexpr int MK_THREADS = (MK_CW + MK_PW) * 32;
constexpr int MK_BOX_ROWS = 16, MK_BOX_COLS = 256;           // row form: two such boxes per slot
constexpr int MK_BOX_BYTES = MK_BOX_ROWS * MK_BOX_COLS * 2;  // 8 KB
constexpr int MK_CBOX_ROWS = 64, MK_CBOX_COLS = 128;         // column form: one box of 64 rows and up to 128 columns per slot
constexpr int MK_SLOT_BYTES = 2 * MK_BOX_BYTES;
constexpr int MK_IN_FLIGHT = 8;                 // slots on their way at once, in the MLP
// and before it, with one row (narrow form) and no more than one band of q/k/v a CTA.  A trip to the L2 queues behind the copies
// on their way to the SM, 2.7 us of them at eight slots, and the phases before the MLP are chains of such trips with little to
// stream: us a layer after 1,000 positions with eight / four here 92.8 / 91.4 (28 query heads, 4 kv heads), 84.5 / 82.7 (32, 2); with
// two bands a CTA 94.4 / 95.4 (32, 8), with four 130.6 / 137.6 (40, 40).
constexpr int MK_FEW_IN_FLIGHT = 4;
constexpr int MK_MAX_ROWS = 4;
constexpr int MK_TC_ROWS = 3;                   // rows from which the tensor-core form runs
constexpr int MK_GROUPS = 4;                    // a slot of weights is the work of one of four groups of four warps
constexpr int MK_MAX_CTAS = 192;                // bounds the number of attention partials
constexpr int MK_SHARED_BYTES = 2688;           // MkShared, behind the area, with two to four rows
constexpr int MK_SHARED_FEW_BYTES = 1536;       // the part of it that one row needs

// The ring, then the area: the activations of a row-form phase (M rows) and what the CTA's own bands make of
// them, or the attention's partials, or the merged heads, or (wide form) the activations of the CTA's share of the
// down-projection.
// Several rows' activations need the larger area, and so does one wide row.  (Wide form, one and two rows: activations that do
// not fit even so, beyond 92 and 44 k-steps, come as a window that is reloaded as the phase moves along.)  A multiple of four
// slots: a weight slot always belongs to the same four warps, so that nobody waits for a slot's next fill before its present
// one has landed.
__host__ __device__ constexpr int mk_slots(int M, bool wide) { return M >= 2 || wide ? 8 : 12; }
__host__ __device__ constexpr int mk_area_bytes(int M, bool wide) { return wide ? 96 * 1024 : M >= 2 ? 88 * 1024 : 33792; }
__host__ __device__ constexpr size_t mk_smem_bytes(int M, bool wide)
{
    return (size_t)mk_slots(M, wide) * MK_SLOT_BYTES + mk_area_bytes(M, wide) + (M >= 2 || wide ? MK_SHARED_BYTES : MK_SHARED_FEW_BYTES);
}
// k-steps of M fp32 activation rows that fit the area beside `own` bytes
__host__ __device__ constexpr int mk_act_window(int M, bool wide, int own) { return (mk_area_bytes(M, wide) - own) / (M * MK_BOX_COLS * 4); }

enum { MKW_Q = 0, MKW_K, MKW_V, MKW_O, MKW_G, MKW_U, MKW_D, MKW_N };
enum { MK_QKV = 0, MK_ATTN = 1, MK_OPROJ = 2, MK_MLP = 3, MK_MAX_PHASES = 5 };
inline int mk_phases(bool wide) { return wide ? 5 : 4; }

// One layer's worth of what the phases need (device array, one entry per layer).
struct MkLayer {
    // per matrix (MKW_*), for passes of one or two rows: [16 rows x 256 columns] boxes, of O and down
    // [64 rows x head_dim or MkCols::box columns] boxes, all without swizzle; then, MKW_N entries on, for
    // passes of three and four rows, which read them with ldmatrix: the same boxes as 64-column blocks with
    // the 128-byte swizzle (view [64][rows][K/64], box {64, 16, 4}), of O and down as 32-column blocks
    // with the 64-byte swizzle (view [32][rows][K/32], box {32, 64, columns / 32})
    CUtensorMap map[14];
    CUtensorMap kmap, vmap;  // the cache as rows of head_dim numbers, boxes of 16 (AttnTma's)
    const bf16 *attn_gain, *mlp_gain;
};

// How the MLP's inner dimension is dealt: contiguous units of `unit` columns (16: a gate/up band; 32 with
// three and four rows) to every CTA, at most `box` columns, one box of the down-projection's columns.
// A box may reach into the next CTA's columns; the activations that meet those are zeros.
// The wide form: a CTA's columns are more than one box, or one activation row does not fit beside twelve slots.  Gate/up deals its bands
// round-robin there and leaves the activation in memory, and the down-projection, a phase of its own, deals
// (block of 128 columns, box of 64 weight rows) pairs evenly.  (Two boxes a CTA, of as many columns as the largest share needs in
// halves, read a tenth too much in slots that are not full: a one-row layer of d_model 7,168, d_ffn 20,480 and 8 kv heads
// after 100 positions 238 us, so 194; of 8,192 and 28,672, its row in windows besides, 369 and 282; two rows of 10,240 and
// 27,648 531 and 374.)
struct MkCols {
    int unit, box;
    bool wide;
};
// k-steps of one row that fit beside the CTA's columns and mk_sums_bytes(1)
constexpr int MK_NARROW_STEPS = (mk_area_bytes(1, false) - MK_CBOX_COLS * 4 - 4096) / (MK_BOX_COLS * 4);
inline MkCols mk_cols(int F, int d, int unit, int n_cta)
{
    const int n = (F + unit - 1) / unit, per = (n + n_cta - 1) / n_cta;
    MkCols c;
    c.unit = unit;
    c.wide = per * unit > MK_CBOX_COLS || (unit == MK_BOX_ROWS && d > MK_NARROW_STEPS * MK_BOX_COLS);
    c.box = c.wide ? MK_CBOX_COLS : per * unit;
    return c;
}

struct MkArgs {
    const MkLayer *layers;       // device
    int layer_begin, layer_end;  // 0-based, [begin, end)
    float *h;                    // residual stream of the pass [rows][d]
    float *h2;                   // [MK_MAX_ROWS][d], zero between launches: what the down-projection has added since h was last whole
    const int *row_slot, *row_pos, *grp_row0, *grp_nrows;
    int n_rows, n_groups;
    kv_t *kc, *vc;               // cache of the first layer [slot][Hkv][S][hd], and what lies between two layers'
    size_t kv_layer;             // (arithmetic: a pointer read from `layers` would be a trip to HBM in every layer)
    float *q_buf;                // [rows][Hq*hd]
    float *act;                  // wide form: [rows][F], the MLP's activation
    float *part_o;               // attention partials, see MkRun
    float2 *part_ml;
    const float2 *rope;
    int d, Hq, Hkv, hd, F, S, n_slots;
    float eps;
    MkCols cols;
    unsigned long long *bar;        // grid barrier counter (monotonic)
    unsigned long long bar_base;    // its value when this launch starts
    int *abort_word;                // nonzero: some CTA gave up
    int *status;
    int short_copy_layer;           // test hook: the layer in which the first CTA's ring waits for bytes that do not come, or -1
    unsigned long long *trace;      // [1 + phases * layers]: CTA 0's clock at the start and after every phase
};

__device__ __forceinline__ unsigned long long ld_acquire_u64(const unsigned long long *p)
{
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ int ld_volatile_i32(const int *p)
{
    int v;
    asm volatile("ld.volatile.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void mk_consumer_sync() { asm volatile("bar.sync 2, %0;" ::"n"(MK_CW * 32) : "memory"); }

// Row form: bands and k-steps.  q/k/v deals whole bands round-robin (144 bands fill 148 SMs well), gate/up
// contiguous bands, because what they make is what the CTA's columns of the down-projection need (wide form: round-robin as well).
struct MkBands {
    int j, end, step, k_steps;
    __device__ void init(int type, const MkArgs &a)
    {
        const int half = a.hd >> 1;
        k_steps = (a.d + MK_BOX_COLS - 1) / MK_BOX_COLS;
        j = blockIdx.x;
        step = gridDim.x;
        if (type == MK_QKV) {
            end = (a.Hq + a.Hkv) * (half / MK_BOX_ROWS) + (a.Hkv * a.hd + 2 * MK_BOX_ROWS - 1) / (2 * MK_BOX_ROWS);
        } else if (a.cols.wide) {
            end = (a.F + MK_BOX_ROWS - 1) / MK_BOX_ROWS;
        } else {
            const int per = a.cols.unit / MK_BOX_ROWS, n = (a.F + a.cols.unit - 1) / a.cols.unit;
            j = (int)(blockIdx.x * (unsigned)n / gridDim.x) * per;
            end = min((int)((blockIdx.x + 1) * (unsigned)n / gridDim.x) * per, (a.F + MK_BOX_ROWS - 1) / MK_BOX_ROWS);
            step = 1;
        }
    }
};
// Descriptor and first row of box `b` (0 or 1) of a band.
__device__ __forceinline__ void mk_band(int type, const MkArgs &a, const MkLayer *L, int band, int b, const CUtensorMap *&map, int &row)
{
    const int half = a.hd >> 1, per_head = half / MK_BOX_ROWS;
    if (type == MK_QKV) {
        const int nq = a.Hq * per_head, nk = a.Hkv * per_head;
        if (band < nq + nk) {
            const bool isq = band < nq;
            const int bb = isq ? band : band - nq;
            map = &L->map[isq ? MKW_Q : MKW_K];
            row = (bb / per_head) * a.hd + (bb % per_head) * MK_BOX_ROWS + b * half;
        } else {
            map = &L->map[MKW_V];
            row = ((band - nq - nk) * 2 + b) * MK_BOX_ROWS;
        }
    } else {
        map = &L->map[b ? MKW_U : MKW_G];
        row = band * MK_BOX_ROWS;
    }
}

// Column form, O-projection: the (head, box of 64 weight rows) pairs laid end to end, head by head, and cut
// into equal contiguous shares [lo, hi); of the wide form's down-projection the same with blocks of 128 columns.
struct MkPairs {
    int boxes, lo, hi;
    __device__ void init(const MkArgs &a, int n)
    {
        boxes = (a.d + MK_CBOX_ROWS - 1) / MK_CBOX_ROWS;
        const unsigned T = (unsigned)n * boxes;
        lo = (int)(blockIdx.x * T / gridDim.x);
        hi = (int)((blockIdx.x + 1) * T / gridDim.x);
    }
};

// Attention: the tiles of 16 positions of all (group, kv head) pairs laid end to end and cut into equal
// contiguous shares, so that every SM reads as much of the cache as the next (with fewer tiles than SMs, one each
// for as many SMs); a run is what a share has of one pair.  The run of pair p in CTA c leaves partial number
// c + p (both only ever grow from one run to the next), for every query vector of the pair.
struct MkRun {
    int t;                          // where it begins in the CTA's share
    int g, hk, tile0, n;            // group, kv head, first tile, tiles
    int row0, nrows, pos0, cache0;  // the group's rows; first cache row of (slot, kv head)
    int nq, n_qblk;                 // query vectors, blocks of eight of them
    int warp0, nsub, item0;         // first warp, warps a block, ring items of the runs beside it
    int part;                       // its partial
};
// What a row of weights of the q/k/v projection becomes: a rotary pair of q or k, or two numbers of v.
struct MkFin {
    float2 cs;      // rotary factors
    size_t off;     // of the first number, the second is `second` behind it
    int second, kind;
};
constexpr int MK_RUNS = 4;
enum { MK_FIN_Q = 0, MK_FIN_K, MK_FIN_V, MK_FIN_NONE };
// The partials of one (row, query head): those of the CTAs [cf, cl], `cell0` plus the CTA's number times mk_part_rows.
struct MkMerge {
    int cf, cl, cell0;
};

// A launch's constants are worked out once: a warp spends some ten cycles an instruction here, so the
// divisions that turn a share into rows and heads held every layer up by 2 us.
struct MkShared {
    uint64_t full[mk_slots(1, false)], empty[mk_slots(1, false)];
    int giving_up, never, go_on;
    int row_slot[MK_MAX_ROWS], row_pos[MK_MAX_ROWS], grp_row0[MK_MAX_ROWS], grp_nrows[MK_MAX_ROWS];  // copies of the row set
    int row_grp[MK_MAX_ROWS];            // group of a row
    int grp_tiles[MK_MAX_ROWS];          // 16-position tiles of a group's prefix
    int att_base[MK_MAX_ROWS + 1];       // tiles x kv heads of the groups before this one
    int att_ctas;                        // CTAs that the tiles are dealt to: none of them goes without
    int att_t0, att_t1;                  // this CTA's share of them
    int att_batch;                       // runs below when they are all of the share and are worked on side by side, or 0
    MkRun runs[MK_RUNS];                 // its first runs
    MkBands bands[2];                    // this CTA's bands of q/k/v and of gate/up
    MkPairs heads;                       // and of the O-projection
    int head0;                           // first head of those
    MkMerge merge[2][MK_MAX_ROWS];       // its first two heads
    float red_rows[MK_MAX_ROWS][MK_CW];  // per-row partial sums of squares
    MkPairs downs;                       // and of the wide form's down-projection
    MkFin fin[MK_BOX_ROWS * MK_MAX_ROWS];  // of the first q/k/v band, [row of the box][activation row]; one row has room for as many
};
static_assert(sizeof(MkShared) <= MK_SHARED_BYTES, "MkShared outgrew its place");
static_assert(offsetof(MkShared, fin) + sizeof(MkFin) * MK_BOX_ROWS <= MK_SHARED_FEW_BYTES, "MkShared outgrew its place");

// A warp's place in the ring: slot and the parity of its present fill.
template <int SLOTS>
struct MkPos {
    int s;
    uint32_t ph;
    __device__ __forceinline__ void skip(int n)   // n < SLOTS
    {
        s += n;
        if (s >= SLOTS) {
            s -= SLOTS;
            ph ^= 1u;
        }
    }
    __device__ __forceinline__ void skip_many(int n)
    {
        const int t = s + n, r = t / SLOTS;
        s = t - r * SLOTS;
        ph ^= (uint32_t)r & 1u;
    }
};

// The run that begins with tile t of a share that ends before `end`.
__device__ __forceinline__ void mk_run_at(const MkArgs &a, const MkShared *sh, int t, int end, MkRun &r)
{
    int g = 0;
#pragma unroll
    for (int i = 1; i < MK_MAX_ROWS; i++)
        if (t >= sh->att_base[i]) g = i;   // (groups without tiles share their successor's base)
    const int tiles = sh->grp_tiles[g], rem = t - sh->att_base[g];
    r.g = g;
    r.hk = rem / tiles;
    r.tile0 = rem - r.hk * tiles;
    r.n = min(tiles - r.tile0, end - t);
    r.row0 = sh->grp_row0[g];
    r.nrows = sh->grp_nrows[g];
    r.pos0 = sh->row_pos[r.row0];
    r.cache0 = (sh->row_slot[r.row0] * a.Hkv + r.hk) * a.S;
    r.nq = r.nrows * (a.Hq / a.Hkv);
    r.n_qblk = (r.nq + 7) / 8;
}
// CTA whose share holds tile t
__device__ __forceinline__ int mk_run_cta(const MkShared *sh, int t)
{
    return (int)((((unsigned)t + 1u) * (unsigned)sh->att_ctas - 1u) / (unsigned)sh->att_base[MK_MAX_ROWS]);
}
// query vectors of a partial
__device__ __forceinline__ int mk_part_rows(const MkArgs &a) { return a.n_rows * (a.Hq / a.Hkv); }

}  // namespace sparsk

#include "sparsk_mega_phases.cuh"
