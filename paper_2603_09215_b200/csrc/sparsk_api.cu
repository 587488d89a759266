// Host side of the SPAR-K decode library: argument checks, the host mirror of the exit
// schedule (which only sizes launches; the device kernels are authoritative), workspace
// carving and the launch sequence of a step.  C ABI declared in include/sparsk.h.
#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <vector>

#include "../../include/sparsk.h"
#include "sparsk_attn.cuh"
#include "sparsk_attn_tc.cuh"
#include "sparsk_common.cuh"
#include "sparsk_gemm.cuh"
#include "sparsk_gemv.cuh"
#include "sparsk_mega.cuh"
#include "sparsk_sample.cuh"
#include "sparsk_step.cuh"

using namespace sparsk;

namespace {

constexpr int MAX_SPLITS = AT_MAX_SPLITS;
constexpr int STAGE_RING = 16;
// Passes of more rows take gate/up units of 128 rows (see build_maps): a CTA's MMA time does not
// depend on the unit's height, so lower units only add CTAs.  First token after 1,024 of the 40-layer
// shape at 256 rows a pass: 51.6 ms with units of 96 rows, 49.8 with 128.
constexpr int GU_EVEN_ROWS = 128;
constexpr uint32_t CTX_MAGIC = 0x5350524bu;  // "SPRK"
constexpr size_t TIME_POOL = 16384;           // event pairs available to the kernel timer
enum { KC_MISC = 0, KC_QKV = 1, KC_ATTN = 2, KC_OPROJ = 3, KC_GATEUP = 4, KC_DOWN = 5, KC_HEAD = 6, KC_MEGA = 7, KC_ALL = 8 };

size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }
int div_up(int a, int b) { return (a + b - 1) / b; }

struct Carve {
    char *base;
    size_t off;
    template <class T>
    T *take(size_t n)
    {
        off = align_up(off, 256);
        T *p = base ? reinterpret_cast<T *>(base + off) : nullptr;
        off += n * sizeof(T);
        return p;
    }
};

}  // namespace

struct TmaPair {
    CUtensorMap m2, m3;
};

struct sparsk_ctx {
    uint32_t magic;
    sparsk_dims dm;
    std::vector<const bf16 *> attn_norm, wq, wk, wv, wo, mlp_norm, w_gate, w_up, w_down, head_norm, head_proj;
    const bf16 *embed;
    cudaStream_t stream;
    int n_sm;
    int cap_rows;  // rows any pass may have
    // workspace
    kv_t *kcache, *vcache;
    float *pend_h;
    int *kv_len, *pend_cnt;
    float2 *rope;
    StepDesc sd;
    int *staged, *tok_dev;
    int *pf_rows;                // row set of a prefill pass: slot and position of every row, the groups, the two counts
    float *h_lo, *h_up;
    float *qbuf;
    float *h_last, *q_last;      // the current rows alone, for the trimmed last layer of the upper pass
    int *last_slot, *last_pos;
    int trim_last;               // 0: never, 1: when it pays (default), 2: whenever there are pending rows
    bf16 *attn_o, *act, *xnorm;
    bf16 *attn_o_lo, *act_lo, *xnorm_lo;  // second bf16 term of the tensor-core path's activations
    float *part_o;
    float2 *part_ml;
    unsigned *attn_ticket;       // device: item counter of the attention kernel (only ever grows)
    unsigned attn_ticket_base;   // host: its value once every launch so far has finished
    int attn_dynamic;            // option: deal attention items by ticket (1, default) or round-robin (0)
    int attn_ctas;               // option: CTAs of the attention kernel (0: as many as fit the SMs)
    // pinned staging ring for the per-step host arrays
    int *stage_host[STAGE_RING];
    int *io_host;                // pinned: [B] tokens in, [B] tokens out, [B] depths out, status (decode_step_host)
    cudaEvent_t stage_ev[STAGE_RING];
    int stage_next;
    // host mirror of per-slot state
    std::vector<int> h_len, h_pend;
    // options
    int pdl, attn_split, gemm_min_rows, gv_ks, gv_r;
    float *dbg_hidden, *dbg_logits;
    // nucleus sampling (off while samp_uniforms is NULL)
    float samp_temperature, samp_top_p;
    const float *samp_uniforms;  // device [max_seqs], read by every decode step
    float *samp_scratch;         // device [max_seqs][Vt + Vs]
    int64_t launches;
    // tensor-core path: TMA descriptors of every weight matrix and of the activation buffers
    // (one per box height 16, 32, ..., 128)
    bool tc_ok;
    std::vector<TmaPair> tm_wq, tm_wk, tm_wv, tm_wo, tm_wg[2], tm_wu[2], tm_wd, tm_head;
    TmaPair tm_x[GM_BOXES], tm_ao[GM_BOXES], tm_act[GM_BOXES];
    int gu_rows[2];              // weight rows per accumulator of a gate/up unit: up to GU_EVEN_ROWS activation rows, beyond
    std::vector<CUtensorMap> tm_kc16, tm_vc16;  // per layer: the cache as rows of head_dim numbers, boxes of 16 rows (attn_warp_tma_kernel)
    int attn_tma, attn_tma_ok;               // option (default 1); the maps above exist
    std::vector<CUtensorMap> tm_kc, tm_vc;  // per layer: the cache viewed as [64][slots * Hkv * S rows][hd / 64], boxes of [64][64][2]
    int attn_stages;                        // K/V ring depth of the warp-per-item attention kernel (2 or 3)
    int attn_tc, attn_tc_min_q;             // tcgen05 attention for blocks of at least this many query vectors
    // persistent layer-range kernel (one to four rows)
    MkLayer *mk_layers;            // device [L]
    unsigned long long *mk_bar;    // device: grid barrier counter; mk_bar_base mirrors its value
    int *mk_abort;                 // device
    float *mk_h2, *mk_act;         // device fp32 [MK_MAX_ROWS][d], [MK_MAX_ROWS][F] (see MkArgs)
    MkCols mk_cols16, mk_cols32;   // how the MLP's columns are dealt to the CTAs, at one and two and at three and four rows
    unsigned long long *mk_trace;  // device [1 + MK_MAX_PHASES L]
    int mk_trace_n;                // entries the last launch wrote
    unsigned long long mk_bar_base;
    int mega, mk_ok, mk_coop, mk_max_rows;
    bool mk_tc_ok;                 // the shape allows the persistent kernel's tensor-core form (3-4 rows)
    // confidence-based exit (dims.conf_modalities != 0): the host drives the step layer by layer
    std::vector<std::vector<int>> h_fill;  // per slot: layer each pending position has been carried to
    int *conf_host;                // pinned arena for the row sets of a step's segments
    size_t conf_host_ints, conf_seg_ints;
    int *conf_rows_dev;            // device: [slot R][pos R][src R][seq R][grp_row0 B][grp_nrows B][n_groups][n_rows]
    int *conf_list_dev;            // device: [rows B][modality B]
    float *conf_ent_dev, *conf_ent_host;  // entropies of a layer's candidates (device, pinned host)
    std::vector<float> conf_trace; // last step: entropy seen at layer l (1-based, < L) by sequence i at [i * L + l], or -1
    float *conf_logits;            // device [B][V] when neither the parity hook nor a sampler lends a buffer
    int inject_timeout;            // test hook: the next persistent launch waits for a barrier count nobody reaches
    int inject_short_copy;         // test hook: the next persistent launch of two layers waits for bytes that do not come
    int64_t route_layers[3];       // layer passes so far by implementation: see sparsk_route_counts
    std::vector<MkLayer> mk_host;
    float *qkv_part;  // fp32 sums of a q/k/v product whose inner dimension is cut across CTAs
    int tc_kb;        // 0: automatic; 1: force one k-block per copy (2-D descriptors)
    int gemm_smem_kb; // shared-memory budget of a tcgen05 GEMM CTA
    int gemm_cps;     // CTAs per SM a split GEMM is cut for (1 or 2; 2 needs a budget that lets two share an SM)
    // optional per-kernel-class timing (events around every launch of one class)
    int cur_class, time_class;
    std::vector<cudaEvent_t> tev;
    std::vector<unsigned char> tev_class;  // class of each bracketed launch
    size_t tev_used;
    char err[512];
};

namespace {

int fail(sparsk_ctx *c, int code, const char *fmt, ...)
{
    if (c) {
        va_list ap;
        va_start(ap, fmt);
        vsnprintf(c->err, sizeof c->err, fmt, ap);
        va_end(ap);
    }
    return code;
}

#define CU(call)                                                                                   \
    do {                                                                                           \
        cudaError_t e_ = (call);                                                                   \
        if (e_ != cudaSuccess)                                                                     \
            return fail(ctx, SPARSK_ECUDA, "%s failed: %s (%s:%d)", #call, cudaGetErrorString(e_), \
                        __FILE__, __LINE__);                                                       \
    } while (0)

bool dims_ok(const sparsk_dims *d)
{
    if (!d) return false;
    if (d->n_layers < 1 || d->d_model < 8 || d->d_model % 8) return false;
    if (d->n_q_heads < 1 || d->n_kv_heads < 1 || d->n_q_heads % d->n_kv_heads) return false;
    if (d->head_dim != 64 && d->head_dim != 128) return false;
    if (d->d_ffn < 8 || d->d_ffn % 8) return false;
    if (d->vocab_text < 1 || d->vocab_speech < 0) return false;
    if (!(d->rms_eps >= 0.f) || !(d->rope_base > 0.f)) return false;
    if (d->exit_layer < 1 || d->exit_layer > d->n_layers) return false;
    if (d->refresh_period < 1 || d->refresh_phase < 0 || d->refresh_phase >= d->refresh_period) return false;
    if (d->text_exit < 0 || d->text_exit > 2) return false;
    if (d->conf_modalities < 0 || d->conf_modalities > 3) return false;
    if (d->conf_modalities && (d->conf_start < 1 || d->conf_start >= d->n_layers || !(d->conf_threshold >= 0.f))) return false;
    if (d->text_period < 0 || (d->text_period > 0 && (d->text_phase < 0 || d->text_phase >= d->text_period))) return false;
    if (d->max_seqs < 1 || d->max_seqs > 1024 || d->max_seq_len < 1) return false;
    if (d->max_pending < 0 || d->prefill_rows < 0) return false;
    return true;
}

// Rows of a prefill pass when the caller leaves the choice to the library.  The GEMMs are bound by the tensor cores
// from 256 rows on (one block of rows), so more rows save no weight traffic, but they give every launch several
// blocks of rows: what a launch costs beyond its products (boundary, ramp, ending) is paid once for all of them,
// the projections with few units need fewer cuts of the inner dimension and so add fewer partials, and
// units that are no multiple of the SMs leave less of the last wave empty.  First token after 1,024: 42.0 ms with
// passes of 256 rows and 33.2 with 1,024 (40-layer shape), 30.9 and 27.0 (28-layer shape); after three times 700
// 63.4 and 54.6.
constexpr int PREFILL_ROWS = 4 * GM_MAX_N;
// Never more rows than the cache has positions.
int prefill_rows_of(const sparsk_dims *d)
{
    return d->prefill_rows > 0 ? d->prefill_rows : (int)std::min<long>(PREFILL_ROWS, std::max<long>(GM_MAX_N, (long)d->max_seqs * d->max_seq_len));
}
long decode_rows_of(const sparsk_dims *d) { return (long)d->max_seqs * (d->max_pending + 1); }
int cap_rows_of(const sparsk_dims *d) { return (int)std::max<long>(decode_rows_of(d), prefill_rows_of(d)); }
// (row, split) pairs the attention partials have room for: every split of a step's rows or of one block of prompt rows.  Passes of more
// prompt rows have fewer splits (run_attn).
size_t part_rows_of(const sparsk_dims *d)
{
    return (size_t)std::max<long>(decode_rows_of(d), std::min(prefill_rows_of(d), GM_MAX_N)) * MAX_SPLITS;
}

// Ints that describe a prefill pass: slot and position of every row, first row and row count of every
// group (one per prompt that takes part), the two counts.
size_t prefill_ints(const sparsk_dims *d) { return 2 * (size_t)cap_rows_of(d) + 2 * (size_t)d->max_seqs + 2; }

// Lays the workspace out; with base == NULL only measures it.
size_t carve(sparsk_ctx *c, const sparsk_dims *d, char *base)
{
    Carve w{base, 0};
    const size_t B = d->max_seqs, S = d->max_seq_len, L = d->n_layers;
    const size_t kvrow = (size_t)d->n_kv_heads * d->head_dim, qrow = (size_t)d->n_q_heads * d->head_dim;
    const size_t R = cap_rows_of(d);
    kv_t *kc = w.take<kv_t>(L * B * S * kvrow);
    kv_t *vc = w.take<kv_t>(L * B * S * kvrow);
    float *ph = w.take<float>(B * (size_t)std::max(1, d->max_pending) * d->d_model);
    int *kl = w.take<int>(B), *pc = w.take<int>(B);
    float2 *rope = w.take<float2>(S * (d->head_dim / 2));
    StepDesc sd;
    sd.slot = w.take<int>(B); sd.modality = w.take<int>(B); sd.depth = w.take<int>(B); sd.lo_pos = w.take<int>(B);
    sd.lo_grp_row0 = w.take<int>(B); sd.lo_grp_nrows = w.take<int>(B);
    sd.up_slot = w.take<int>(R); sd.up_pos = w.take<int>(R); sd.up_src = w.take<int>(R);
    sd.up_grp_row0 = w.take<int>(B); sd.up_grp_nrows = w.take<int>(B); sd.cur_row = w.take<int>(B);
    sd.list_seq = w.take<int>(4 * B); sd.list_row = w.take<int>(4 * B);
    sd.counts = w.take<int>(8);
    sd.argmax = w.take<unsigned long long>(B);
    int *staged = w.take<int>(3 * B), *tok = w.take<int>(B);
    int *pfr = w.take<int>(prefill_ints(d));
    float *hlo = w.take<float>(B * d->d_model), *hup = w.take<float>(R * d->d_model);
    float *q = w.take<float>(R * qrow);
    int *crows = nullptr, *clist = nullptr;
    float *cent = nullptr, *clog = nullptr;
    if (d->conf_modalities) {
        crows = w.take<int>(4 * R + 2 * B + 2);
        clist = w.take<int>(2 * B);
        cent = w.take<float>(B);
        clog = w.take<float>(B * ((size_t)d->vocab_text + d->vocab_speech));
    }
    float *hlast = w.take<float>(B * d->d_model), *qlast = w.take<float>(B * qrow);
    int *lslot = w.take<int>(B), *lpos = w.take<int>(B);
    bf16 *ao = w.take<bf16>(R * qrow), *act = w.take<bf16>(R * d->d_ffn);
    bf16 *xn = w.take<bf16>(R * d->d_model);
    bf16 *aol = w.take<bf16>(R * qrow), *actl = w.take<bf16>(R * d->d_ffn), *xnl = w.take<bf16>(R * d->d_model);
    float *qp = w.take<float>(R * (qrow + 2 * kvrow));
    MkLayer *mkl = w.take<MkLayer>(L);
    unsigned long long *mkb = w.take<unsigned long long>(1);
    int *mka = w.take<int>(1);
    unsigned *atk = w.take<unsigned>(1);
    float *mkh2 = w.take<float>((size_t)MK_MAX_ROWS * d->d_model), *mkact = w.take<float>((size_t)MK_MAX_ROWS * d->d_ffn);
    unsigned long long *mkt = w.take<unsigned long long>(1 + MK_MAX_PHASES * L);
    // attention partials: of the launches, and of the persistent kernel (see MkRun)
    const size_t runs = (size_t)MK_MAX_CTAS + (size_t)MK_MAX_ROWS * d->n_kv_heads;
    const size_t cells = std::max<size_t>(std::max(R, part_rows_of(d)) * d->n_q_heads, runs * MK_MAX_ROWS * (d->n_q_heads / d->n_kv_heads));
    float *po = w.take<float>(cells * d->head_dim);
    float2 *pml = w.take<float2>(cells);
    if (c) {
        c->kcache = kc; c->vcache = vc; c->pend_h = ph; c->kv_len = kl; c->pend_cnt = pc; c->rope = rope;
        c->sd = sd; c->staged = staged; c->tok_dev = tok;
        c->pf_rows = pfr;
        c->conf_rows_dev = crows; c->conf_list_dev = clist; c->conf_ent_dev = cent; c->conf_logits = clog;
        c->h_last = hlast; c->q_last = qlast; c->last_slot = lslot; c->last_pos = lpos;
        c->h_lo = hlo; c->h_up = hup; c->qbuf = q; c->attn_o = ao; c->act = act; c->xnorm = xn; c->qkv_part = qp;
        c->attn_o_lo = aol; c->act_lo = actl; c->xnorm_lo = xnl;
        c->mk_layers = mkl; c->mk_bar = mkb; c->mk_abort = mka; c->mk_h2 = mkh2; c->mk_act = mkact; c->mk_trace = mkt;
        c->part_o = po; c->part_ml = pml; c->attn_ticket = atk;
    }
    return align_up(w.off, 256);
}

// cluster: CTAs per cluster along x
template <class... KArgs, class... Args>
cudaError_t launch_clusters(sparsk_ctx *c, int cluster, void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, Args... args)
{
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof cfg);
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = c->stream;
    cudaLaunchAttribute attr[2];
    cfg.attrs = attr;
    if (c->pdl) {
        attr[cfg.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[cfg.numAttrs++].val.programmaticStreamSerializationAllowed = 1;
    }
    if (cluster > 1) {
        attr[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
        attr[cfg.numAttrs].val.clusterDim.x = cluster;
        attr[cfg.numAttrs].val.clusterDim.y = 1;
        attr[cfg.numAttrs++].val.clusterDim.z = 1;
    }
    c->launches++;
    const bool timed = ((c->time_class == c->cur_class && c->time_class != KC_MISC) || c->time_class == KC_ALL) &&
                       c->tev_used + 2 <= c->tev.size();
    if (timed) {
        c->tev_class[c->tev_used / 2] = (unsigned char)c->cur_class;
        cudaEventRecord(c->tev[c->tev_used++], c->stream);
    }
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, KArgs(args)...);
    if (timed) cudaEventRecord(c->tev[c->tev_used++], c->stream);
    return e;
}

template <class... KArgs, class... Args>
cudaError_t launch(sparsk_ctx *c, void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, Args... args)
{
    return launch_clusters(c, 1, kern, grid, block, smem, args...);
}

// ---------------------------------------------------------------- GEMV dispatch
struct GvPlan {
    int ks, grid_x;
};

GvPlan plan_gemv(const sparsk_ctx *c, int n_groups, int K)
{
    const int chunks = (K + 255) / 256;
    int best_ks = 1;
    double best = 1e30;
    for (int ks = 1; ks <= GV_WARPS; ks *= 2) {
        if (ks > 1 && ks > chunks) break;
        const long T = (long)c->n_sm * (GV_WARPS / ks);
        const long iters = (n_groups + T - 1) / T;
        const double cost = (double)iters * ((chunks + ks - 1) / ks + 3.0);
        if (cost < best - 1e-9) {
            best = cost;
            best_ks = ks;
        }
    }
    if (c->gv_ks > 0) best_ks = c->gv_ks;
    GvPlan p;
    p.ks = best_ks;
    p.grid_x = std::min(c->n_sm, n_groups);
    if (p.grid_x < 1) p.grid_x = 1;
    return p;
}

template <class Op, int R, int M, bool NORM>
cudaError_t launch_gemv_inst(sparsk_ctx *c, const Op &op, GvIn in, int n_groups)
{
    static PerDevice<bool> attr_done;
    bool &attr_set = attr_done.here();
    auto kern = gemv_kernel<Op, R, M, NORM>;
    if (!attr_set) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
        if (e != cudaSuccess) return e;
        attr_set = true;
    }
    const GvPlan p = plan_gemv(c, n_groups, in.K);
    in.ks = p.ks;
    const size_t smem = align_up((size_t)M * in.K * 2, 16) + (size_t)2 * GV_WARPS * R * M * sizeof(float);
    if (smem > 200 * 1024) return cudaErrorInvalidValue;
    const int passes = (M == GV_MC) ? (in.n_rows + GV_MC - 1) / GV_MC : 1;
    return launch(c, kern, dim3(p.grid_x, passes), dim3(GV_THREADS), smem, op, in);
}

// M template: 1, 2 or 4 (three rows run as four with one masked).
#define GV_DISPATCH_M(OPT, RR, NORM, op, in, ng)                                    \
    ((in).n_rows == 1   ? launch_gemv_inst<OPT<RR>, RR, 1, NORM>(c, op, in, ng)     \
     : (in).n_rows == 2 ? launch_gemv_inst<OPT<RR>, RR, 2, NORM>(c, op, in, ng)     \
                        : launch_gemv_inst<OPT<RR>, RR, 4, NORM>(c, op, in, ng))

int pick_r(const sparsk_ctx *c, int n_rows, bool paired)
{
    if (c->gv_r > 0) return (paired && c->gv_r < 2) ? 2 : c->gv_r;
    if (n_rows >= 3) return 4;
    return 2;
}

struct PromptGroup {
    int rows, len;  // of a prompt pass's group: rows, and positions the last of them attends to
};
struct RowSet {
    const int *slot, *pos, *grp_row0, *grp_nrows, *n_groups, *n_rows_dev;
    int n_rows;     // host count (sizes the launches)
    int n_groups_h; // host count
    int max_grp_rows;
    int max_len;    // longest prefix any row attends to (host)
    int n_big;      // groups with at least attn_tc_min_q query vectors per kv head (0: not counted, assume all)
    const float *q; // the rows' queries if they are not the context's query buffer (NULL: they are)
    long sum_len;   // total of the groups' prefix lengths (host; 0: unknown)
    bool rows_late; // the arrays are written by a kernel that may still run when the pass's kernels start
    const PromptGroup *prompt;      // prompt passes: the groups (host), else NULL
    mutable int splits_tc, splits_warp;  // prompt passes: even_splits' answers for the two attention kernels, once asked (0 before)
};

cudaError_t run_qkv(sparsk_ctx *c, int layer, const float *h, const RowSet &rs)
{
    const sparsk_dims &d = c->dm;
    const int li = layer - 1;
    GvIn in{};
    in.h = h; in.gain = c->attn_norm[li]; in.eps = d.rms_eps; in.K = d.d_model; in.n_rows = rs.n_rows;
    const size_t lstride = (size_t)d.max_seqs * d.n_kv_heads * d.max_seq_len * d.head_dim;
    const int R = pick_r(c, rs.n_rows, true);
#define QKV_CASE(RR)                                                                                   \
    {                                                                                                  \
        QkvOp<RR> op;                                                                                  \
        op.wq = c->wq[li]; op.wk = c->wk[li]; op.wv = c->wv[li]; op.q_out = c->qbuf;                   \
        op.kc = c->kcache + li * lstride; op.vc = c->vcache + li * lstride; op.rope = c->rope;         \
        op.row_slot = rs.slot; op.row_pos = rs.pos; op.d = d.d_model; op.Hq = d.n_q_heads;             \
        op.Hkv = d.n_kv_heads; op.hd = d.head_dim; op.S = d.max_seq_len;                               \
        const int P = RR / 2;                                                                          \
        const int ng = (d.n_q_heads + d.n_kv_heads) * (d.head_dim / 2) / P + d.n_kv_heads * d.head_dim / RR; \
        return GV_DISPATCH_M(QkvOp, RR, true, op, in, ng);                                             \
    }
    if (R == 4) QKV_CASE(4) else QKV_CASE(2)
#undef QKV_CASE
}

cudaError_t run_resid(sparsk_ctx *c, const bf16 *w, const bf16 *x, float *h, int K, int n_out, int n_rows)
{
    GvIn in{};
    in.x = x; in.K = K; in.n_rows = n_rows;
    int R = c->gv_r > 0 ? c->gv_r : (n_rows >= 3 ? 4 : 2);
#define RES_CASE(RR)                                            \
    {                                                           \
        ResidOp<RR> op;                                         \
        op.w = w; op.h = h; op.K = K; op.n_out = n_out;         \
        const int ng = (n_out + RR - 1) / RR;                   \
        return GV_DISPATCH_M(ResidOp, RR, false, op, in, ng);   \
    }
    if (R == 4) RES_CASE(4) else if (R == 2) RES_CASE(2) else RES_CASE(1)
#undef RES_CASE
}

cudaError_t run_gateup(sparsk_ctx *c, int layer, const float *h, int n_rows)
{
    const sparsk_dims &d = c->dm;
    const int li = layer - 1;
    GvIn in{};
    in.h = h; in.gain = c->mlp_norm[li]; in.eps = d.rms_eps; in.K = d.d_model; in.n_rows = n_rows;
    const int R = pick_r(c, n_rows, true);
#define GU_CASE(RR)                                                              \
    {                                                                            \
        GateUpOp<RR> op;                                                         \
        op.wg = c->w_gate[li]; op.wu = c->w_up[li]; op.u = c->act;               \
        op.d = d.d_model; op.F = d.d_ffn;                                        \
        const int P = RR / 2;                                                    \
        const int ng = (d.d_ffn + P - 1) / P;                                    \
        return GV_DISPATCH_M(GateUpOp, RR, true, op, in, ng);                    \
    }
    if (R == 4) GU_CASE(4) else GU_CASE(2)
#undef GU_CASE
}

// Where the heads leave their logits: the parity hook's buffer, else the sampler's, else nowhere.
float *head_logits(const sparsk_ctx *c)
{
    return c->dbg_logits ? c->dbg_logits : (c->samp_uniforms ? c->samp_scratch : c->conf_logits);
}

bool use_tc(const sparsk_ctx *c, int n_rows);
cudaError_t run_head_tc(sparsk_ctx *c, int layer, const float *h, int list, int n_rows);

// Head of `layer` over list `l` (0 early/text, 1 early/speech, 2 full/text, 3 full/speech).
cudaError_t run_head(sparsk_ctx *c, int layer, const float *h, int list, int n_rows)
{
    const sparsk_dims &d = c->dm;
    const int li = layer - 1, B = d.max_seqs;
    GvIn in{};
    in.h = h; in.gain = c->head_norm[li]; in.eps = d.rms_eps; in.K = d.d_model; in.n_rows = n_rows;
    in.row_idx = c->sd.list_row + (size_t)list * B;
    const int speech = list & 1;
    if (use_tc(c, n_rows)) return run_head_tc(c, layer, h, list, n_rows);
    const int R = c->gv_r > 0 ? c->gv_r : 4;
    struct ClassScope {
        sparsk_ctx *c;
        ~ClassScope() { c->cur_class = KC_MISC; }
    } scope{c};
    c->cur_class = KC_HEAD;
#define HD_CASE(RR)                                                                              \
    {                                                                                            \
        HeadOp<RR> op;                                                                           \
        op.w = c->head_proj[li]; op.seq_of_row = c->sd.list_seq + (size_t)list * B;              \
        op.argmax = c->sd.argmax; op.logits = head_logits(c); op.d = d.d_model;                   \
        op.lo = speech ? d.vocab_text : 0; op.hi = speech ? d.vocab_text + d.vocab_speech : d.vocab_text; \
        op.V = d.vocab_text + d.vocab_speech;                                                    \
        const int ng = (op.hi - op.lo + RR - 1) / RR;                                            \
        return GV_DISPATCH_M(HeadOp, RR, true, op, in, ng);                                      \
    }
    if (R == 4) HD_CASE(4) else if (R == 2) HD_CASE(2) else HD_CASE(1)
#undef HD_CASE
}


// Splits of a prompt pass whose groups are uneven.  The plans below take every group for the largest, in rows and in positions: where a few
// rows behind a long prefix share a pass with many rows of a short one, that fills the machine on paper with one split, and one
// worker is left with the whole prefix.  Here a plan's time is estimated, in positions of one item: whole rounds of its long items (or
// the mean load, where that is more), `setup` for each round of items, `merge` for each split; `now` splits stay unless more of them
// are better by a sixth.  us a layer, passes of 256 rows without this / one pass without / with it: two rows behind 60,000
// positions and 700 without, 16 heads and kv heads of 64 739 / 2,243 / 334, 32 and 8 of 64 1,872 / 2,373 / 463; eight rows behind
// 60,000 and three times 300, 28 and 4 heads of 128 1,104 / 1,842 / 946.
int even_splits(const RowSet &rs, int q_min, int q_max, int G, int Hkv, int block, int workers, int tile, double setup, double merge,
                int now, int max_splits)
{
    auto time = [&](int n) {
        const int len = div_up(div_up(rs.max_len, n), tile) * tile;
        double full = 0, items = 0, work = 0;
        for (int g = 0; g < rs.n_groups_h; g++) {
            const int q = rs.prompt[g].rows * G;
            if (q < q_min || q > q_max) continue;
            const double blocks = (double)div_up(q, block) * Hkv;
            full += blocks * ((rs.prompt[g].len + len / 2) / len);
            items += blocks * div_up(rs.prompt[g].len, len);
            work += blocks * rs.prompt[g].len;
        }
        return std::max(std::ceil(full / workers) * len, work / workers) + std::ceil(items / workers) * setup + n * merge;
    };
    const double at_first = time(now);
    double best = at_first;
    int n_best = now;
    for (int n = now + 1; n <= max_splits && div_up(rs.max_len, n) >= 8 * tile; n++) {
        const double t = time(n);
        if (t < best) {
            best = t;
            n_best = n;
        }
    }
    return best < at_first * 5 / 6 ? n_best : now;
}

cudaError_t run_attn(sparsk_ctx *c, int layer, const RowSet &rs)
{
    const sparsk_dims &d = c->dm;
    const int G = d.n_q_heads / d.n_kv_heads;
    const size_t lstride = (size_t)d.max_seqs * d.n_kv_heads * d.max_seq_len * d.head_dim;
    AttnArgs a{};
    a.q = nullptr;
    a.q32 = rs.q ? rs.q : c->qbuf;
    a.kc = c->kcache + (layer - 1) * lstride;
    a.vc = c->vcache + (layer - 1) * lstride;
    a.grp_row0 = rs.grp_row0; a.grp_nrows = rs.grp_nrows; a.row_slot = rs.slot; a.row_pos = rs.pos;
    a.n_groups = rs.n_groups;
    a.part_o = c->part_o; a.part_ml = c->part_ml; a.out = c->attn_o; a.out_lo = c->attn_o_lo;
    a.Hq = d.n_q_heads; a.Hkv = d.n_kv_heads; a.S = d.max_seq_len;
    a.n_slots = d.max_seqs;
    a.n_rows = rs.n_rows;
    a.nq_min = 0;
    a.nq_max = 1 << 30;
    a.rows_early = !rs.rows_late;
    cudaError_t e;
    const int max_splits = (int)std::min<size_t>(AT_MAX_SPLITS, std::max<size_t>(1, part_rows_of(&d) / rs.n_rows));
    const bool blocks_tc = c->attn_tc && c->tc_ok && d.head_dim == TA_HD && rs.max_grp_rows * G >= c->attn_tc_min_q;
    // groups the tcgen05 kernel takes (the host knows every group's row count) and the rest
    const int n_big = blocks_tc ? (rs.n_big > 0 ? rs.n_big : rs.n_groups_h) : 0;
    const int n_small = rs.n_groups_h - n_big;
    const int warp_ctas = c->attn_ctas > 0 ? c->attn_ctas : c->n_sm * attn_warp_ctas_per_sm(d.head_dim, c->attn_stages);
    const int small_rows = blocks_tc ? std::max(1, std::min(rs.max_grp_rows, (c->attn_tc_min_q - 1) / G)) : rs.max_grp_rows;
    const bool tma = c->attn_tma && c->attn_tma_ok;
    a.table = tma && rs.n_groups_h <= AT_TABLE;
    AttnPlan pl = attn_plan(warp_ctas * AW_WARPS, blocks_tc ? std::max(1, n_small) : rs.n_groups_h, small_rows, G,
                            d.n_kv_heads, rs.max_len, c->attn_split, blocks_tc ? 0 : rs.sum_len, a.table);
    if (pl.n_splits > max_splits) {
        pl.split_len = div_up(div_up(rs.max_len, max_splits), AT_TP) * AT_TP;
        pl.n_splits = div_up(rs.max_len, pl.split_len);
    }
    // bytes of a split's partials, written and read, in us
    const double merge_us = (double)rs.n_rows * d.n_q_heads * d.head_dim * 8 / 5e6;
    if (rs.prompt && c->attn_split <= 0 && (!blocks_tc || n_small > 0)) {
        if (!rs.splits_warp)  // (16 positions are 0.5 us, an item's set-up four tiles)
            rs.splits_warp = even_splits(rs, 0, blocks_tc ? c->attn_tc_min_q - 1 : 1 << 30, G, d.n_kv_heads, 16, warp_ctas * AW_WARPS, AT_TP,
                                         4 * AT_TP, merge_us * 32, pl.n_splits, max_splits);
        if (rs.splits_warp > pl.n_splits) {
            pl.split_len = div_up(div_up(rs.max_len, rs.splits_warp), AT_TP) * AT_TP;
            pl.n_splits = div_up(rs.max_len, pl.split_len);
        }
    }
    if (blocks_tc) {
        // Groups with many query vectors per kv head go to the tcgen05 kernel (one CTA per SM, tiles
        // of 64 positions), the others to the mma.sync kernel; both launches cover all groups, a CTA
        // leaves at once if its group belongs to the other, and both use one split plan so that the
        // merge finds every partial where it expects it.
        static PerDevice<bool> ready_dev;
        bool &ready = ready_dev.here();
        if (!ready) {
            if ((e = cudaFuncSetAttribute(attn_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, TA_SMEM)) != cudaSuccess) return e;
            ready = true;
        }
        // The tcgen05 kernel wants few, long splits (about one CTA per SM from the big groups alone,
        // its set-up is worth a few tiles), the other kernel many short ones: the first kernel's
        // split is `mult` of the second's, and it marks the partial slots in between as empty.  Without
        // groups for the second kernel the partials lie side by side, and a single one is finished
        // by the kernel itself, without a merge: the merge of a pass of 256 prompt rows read up to sixteen
        // slots per row and head for its one or two partials, 13.8 us a layer (ragged prompts over
        // the 28-layer shape 206 -> 193 ms, 1,024 tokens over the 40-layer shape 44.9 -> 43.3).
        const int big_ctas = std::max(1, n_big * div_up(rs.max_grp_rows * G, TA_QB) * d.n_kv_heads);
        const int tiles = std::max(1, div_up(rs.max_len, TA_NT));
        int s_tc = 1;
        {   // the split count whose CTAs fill whole waves of one CTA per SM best (at least 8 tiles each)
            double best = -1.0;
            const int s_max = std::max(1, std::min(max_splits, tiles / 8));
            for (int sc = 1; sc <= s_max; sc++) {
                const long n = (long)big_ctas * sc, waves = (n + c->n_sm - 1) / c->n_sm;
                const double eff = (double)n / (double)(waves * c->n_sm);
                const double score = eff * (waves >= 2 ? 1.0 : 0.9);  // a second wave evens out ragged lengths
                if (score > best + 1e-9) {
                    best = score;
                    s_tc = sc;
                }
                if (waves >= 2 && eff >= 0.9) break;
            }
        }
        if (c->attn_split > 0) s_tc = pl.n_splits;
        s_tc = std::min(s_tc, max_splits);
        if (rs.prompt && c->attn_split <= 0) {  // (64 positions are 0.4 us, a set-up four tiles)
            if (!rs.splits_tc)
                rs.splits_tc = even_splits(rs, c->attn_tc_min_q, 1 << 30, G, d.n_kv_heads, TA_QB, c->n_sm, TA_NT, 4 * TA_NT, merge_us * 160, s_tc,
                                           max_splits);
            s_tc = rs.splits_tc;
        }
        const int mult = n_small > 0 ? std::max(1, std::min(max_splits / s_tc, div_up(pl.n_splits, s_tc))) : 1;
        const int small_len = div_up(div_up(rs.max_len, s_tc * mult), TA_NT) * TA_NT;
        pl.split_len = small_len;
        pl.n_splits = std::max(1, div_up(rs.max_len, small_len));
        AttnTcArgs ta;
        ta.a = a;
        ta.a.n_qblk = div_up(rs.max_grp_rows * G, TA_QB);
        ta.a.split_len = small_len * mult;
        ta.a.n_splits = pl.n_splits;
        ta.a.nq_min = c->attn_tc_min_q;
        ta.split_mult = mult;
        ta.direct = pl.n_splits == 1 && n_small == 0;
        ta.status = c->sd.counts + CNT_STATUS;
        const int n_splits_tc = std::max(1, div_up(rs.max_len, small_len * mult));
        dim3 grid(rs.n_groups_h * ta.a.n_qblk, d.n_kv_heads, n_splits_tc);
        e = launch(c, attn_tc_kernel, grid, dim3(TA_THREADS), (size_t)TA_SMEM, c->tm_kc[layer - 1], c->tm_vc[layer - 1], ta);
        if (e != cudaSuccess || ta.direct) return e;
        a.nq_max = c->attn_tc_min_q - 1;
    }
    a.n_qblk = blocks_tc ? div_up(std::min(rs.max_grp_rows * G, c->attn_tc_min_q - 1), 16) : pl.n_qblk;
    a.split_len = pl.split_len;
    a.n_splits = pl.n_splits;
    a.max_groups = rs.n_groups_h;
    if (!blocks_tc || (c->attn_tc_min_q > 1 && n_small > 0)) {
        // every group is in the item space (the kernel skips those the other kernel takes)
        const long n_items = (long)rs.n_groups_h * a.n_qblk * d.n_kv_heads * a.n_splits;
        int warps = AW_WARPS;
        AttnWarpFn fn = nullptr;
        AttnWarpTmaFn fn_tma = nullptr;
        e = tma ? attn_warp_tma_fn(d.head_dim, c->attn_stages, &fn_tma, &warps) : attn_warp_fn(d.head_dim, c->attn_stages, &fn);
        if (e != cudaSuccess) return e;
        const int grid = (int)std::max<long>(1, std::min<long>(warp_ctas, (n_items + warps - 1) / warps));
        if (c->attn_dynamic && n_items < (1L << 31)) {
            a.ticket = c->attn_ticket;
            a.ticket_base = c->attn_ticket_base;
        }
        if (tma)
            e = launch(c, fn_tma, dim3(grid), dim3(warps * 32), attn_warp_tma_bytes(d.head_dim, c->attn_stages, warps),
                       c->tm_kc16[layer - 1], c->tm_vc16[layer - 1], a, c->sd.counts + CNT_STATUS);
        else
            e = launch(c, fn, dim3(grid), dim3(warps * 32), AW_WARPS * attn_warp_bytes(d.head_dim, c->attn_stages), a);
        if (e != cudaSuccess) return e;
        // the items beyond the warps' first ones are drawn once each, and every warp draws one
        // ticket beyond its last item
        if (a.ticket && n_items > (long)grid * warps) c->attn_ticket_base += (unsigned)n_items;
    }
    dim3 grid;
    const AttnMergeFn merge = attn_merge_fn(d.head_dim, a.n_splits, rs.n_rows, d.n_q_heads, &grid);
    return launch(c, merge, grid, dim3(MG_THREADS), 0, a, rs.n_rows_dev);
}

// ---------------------------------------------------------------- tensor-core dispatch
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// Descriptors of a row-major 16-bit matrix [rows][cols], 128-byte swizzle, zero fill outside:
// m2 reads boxes of [box_rows][64]; m3 (only when cols is a multiple of 64) views the matrix as
// [64][rows][cols/64] and reads [box_rows] rows of two consecutive 64-element blocks at once.
bool encode_maps(EncodeTiledFn fn, TmaPair *m, const void *base, size_t rows, size_t cols, int box_rows,
                 CUtensorMapDataType dtype)
{
    memset(m, 0, sizeof *m);
    if (!base) return true;
    const cuuint32_t es[3] = {1, 1, 1};
    {
        const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
        const cuuint64_t strides[1] = {(cuuint64_t)cols * 2};
        const cuuint32_t box[2] = {(cuuint32_t)GM_BK, (cuuint32_t)box_rows};
        if (fn(&m->m2, dtype, 2, const_cast<void *>(base), dims, strides, box, es,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return false;
    }
    if (cols % GM_BK == 0) {
        const cuuint64_t dims[3] = {(cuuint64_t)GM_BK, (cuuint64_t)rows, (cuuint64_t)(cols / GM_BK)};
        const cuuint64_t strides[2] = {(cuuint64_t)cols * 2, (cuuint64_t)GM_BK * 2};
        const cuuint32_t box[3] = {(cuuint32_t)GM_BK, (cuuint32_t)box_rows, 2};
        if (fn(&m->m3, dtype, 3, const_cast<void *>(base), dims, strides, box, es,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return false;
    }
    return true;
}

// Descriptors of an operand of the tcgen05 GEMMs: a row-major bf16 matrix, or (lo) the two planes
// of an activation matrix: a box carries the same rows of every plane, the lo tile behind the hi
// tile.  m2 takes one 64-element block per copy (view [cols][rows][plane]), m3 two (view
// [64][rows][plane][cols/64]).
bool encode_gemm_maps(EncodeTiledFn fn, TmaPair *m, const bf16 *hi, const bf16 *lo, size_t rows, size_t cols, int box_rows)
{
    memset(m, 0, sizeof *m);
    if (!hi) return true;
    const cuuint64_t planes = lo ? 2 : 1, row = (cuuint64_t)cols * 2, plane = lo ? (cuuint64_t)((const char *)lo - (const char *)hi) : row * rows;
    const cuuint32_t es[4] = {1, 1, 1, 1}, box_planes = (cuuint32_t)planes;
    {
        const cuuint64_t dims[3] = {(cuuint64_t)cols, (cuuint64_t)rows, planes}, strides[2] = {row, plane};
        const cuuint32_t box[3] = {(cuuint32_t)GM_BK, (cuuint32_t)box_rows, box_planes};
        if (fn(&m->m2, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<bf16 *>(hi), dims, strides, box, es,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return false;
    }
    if (cols % GM_BK == 0) {
        const cuuint64_t dims[4] = {(cuuint64_t)GM_BK, (cuuint64_t)rows, planes, (cuuint64_t)(cols / GM_BK)};
        const cuuint64_t strides[3] = {row, plane, (cuuint64_t)GM_BK * 2};
        const cuuint32_t box[4] = {(cuuint32_t)GM_BK, (cuuint32_t)box_rows, box_planes, 2};
        if (fn(&m->m3, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<bf16 *>(hi), dims, strides, box, es,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return false;
    }
    return true;
}

bool build_maps(sparsk_ctx *c)
{
    const sparsk_dims &d = c->dm;
    void *fp = nullptr;
    cudaDriverEntryPointQueryResult qr;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fp, cudaEnableDefault, &qr) != cudaSuccess || !fp ||
        qr != cudaDriverEntryPointSuccess)
        return false;
    EncodeTiledFn fn = (EncodeTiledFn)fp;
    const int L = d.n_layers, V = d.vocab_text + d.vocab_speech;
    const size_t qd = (size_t)d.n_q_heads * d.head_dim, kd = (size_t)d.n_kv_heads * d.head_dim;
    bool ok = true;
    auto fill = [&](std::vector<TmaPair> &v, const std::vector<const bf16 *> &w, size_t rows, size_t cols, int box) {
        v.resize(L);
        for (int l = 0; l < L; l++) ok = ok && encode_gemm_maps(fn, &v[l], w[l], nullptr, rows, cols, box);
    };
    fill(c->tm_wq, c->wq, qd, d.d_model, 2 * GM_BM); fill(c->tm_wk, c->wk, kd, d.d_model, 2 * GM_BM);
    fill(c->tm_wv, c->wv, kd, d.d_model, 2 * GM_BM); fill(c->tm_wo, c->wo, d.d_model, qd, 2 * GM_BM);
    // gate/up unit height: dealt evenly to the SMs, or, where the MMAs and not the weight stream take
    // the time, what an MMA covers, the full 128
    c->gu_rows[0] = gateup_unit_rows(d.d_ffn, c->n_sm);
    c->gu_rows[1] = GM_BM;
    for (int t = 0; t < 2; t++) {
        fill(c->tm_wg[t], c->w_gate, d.d_ffn, d.d_model, c->gu_rows[t]);
        fill(c->tm_wu[t], c->w_up, d.d_ffn, d.d_model, c->gu_rows[t]);
    }
    fill(c->tm_wd, c->w_down, d.d_model, d.d_ffn, 2 * GM_BM); fill(c->tm_head, c->head_proj, V, d.d_model, 2 * GM_BM);
    if (d.head_dim == 64 || d.head_dim == 128) {
        const size_t lstride = (size_t)d.max_seqs * d.n_kv_heads * d.max_seq_len * d.head_dim;
        const size_t rows = (size_t)d.max_seqs * d.n_kv_heads * d.max_seq_len;
        c->tm_kc16.resize(L);
        c->tm_vc16.resize(L);
        bool ok16 = rows < (1ull << 31);
        for (int l = 0; l < L && ok16; l++) {
            TmaPair t;
            ok16 = ok16 && encode_maps(fn, &t, c->kcache + l * lstride, rows, d.head_dim, AT_TP, CU_TENSOR_MAP_DATA_TYPE_FLOAT16);
            c->tm_kc16[l] = d.head_dim == 128 ? t.m3 : t.m2;
            ok16 = ok16 && encode_maps(fn, &t, c->vcache + l * lstride, rows, d.head_dim, AT_TP, CU_TENSOR_MAP_DATA_TYPE_FLOAT16);
            c->tm_vc16[l] = d.head_dim == 128 ? t.m3 : t.m2;
        }
        c->attn_tma_ok = ok16 ? 1 : 0;
    }
    if (d.head_dim == TA_HD) {
        const size_t lstride = (size_t)d.max_seqs * d.n_kv_heads * d.max_seq_len * d.head_dim;
        c->tm_kc.resize(L);
        c->tm_vc.resize(L);
        for (int l = 0; l < L && ok; l++) {
            TmaPair t;
            ok = ok && encode_maps(fn, &t, c->kcache + l * lstride, (size_t)d.max_seqs * d.n_kv_heads * d.max_seq_len, d.head_dim, TA_NT,
                                   CU_TENSOR_MAP_DATA_TYPE_FLOAT16);
            c->tm_kc[l] = t.m3;
            ok = ok && encode_maps(fn, &t, c->vcache + l * lstride, (size_t)d.max_seqs * d.n_kv_heads * d.max_seq_len, d.head_dim, TA_NT,
                                   CU_TENSOR_MAP_DATA_TYPE_FLOAT16);
            c->tm_vc[l] = t.m3;
        }
    }
    for (int b = 0; b < GM_BOXES; b++) {
        const int box = 16 * (b + 1);
        ok = ok && encode_gemm_maps(fn, &c->tm_x[b], c->xnorm, c->xnorm_lo, c->cap_rows, d.d_model, box);
        ok = ok && encode_gemm_maps(fn, &c->tm_ao[b], c->attn_o, c->attn_o_lo, c->cap_rows, qd, box);
        ok = ok && encode_gemm_maps(fn, &c->tm_act[b], c->act, c->act_lo, c->cap_rows, d.d_ffn, box);
    }
    return ok;
}

// Activation rows per copy: as many as a CTA takes, in steps of 16 (a copy of rows that do not exist
// costs L2 traffic and ring space: 70 rows in a 128-row box left room for one k-block per copy).
int box_index(int rows_per_cta) { return (rows_per_cta + 15) / 16 - 1; }

template <class Epi, bool DUO>
cudaError_t launch_gemm_inst(sparsk_ctx *c, const TmaPair &a0, const TmaPair &a1, const TmaPair &a2, const TmaPair *b_maps,
                        GemmArgs g, const Epi &epi)
{
    static PerDevice<bool> attr_done;
    bool &attr_set = attr_done.here();
    constexpr int SMEM_BUDGET = 220 * 1024;
    auto kern = wsgemm_kernel<Epi, DUO>;
    if (!attr_set) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BUDGET);
        if (e != cudaSuccess) return e;
        attr_set = true;
    }
    const int bi = box_index(DUO ? (std::min(g.m_rows, GM_MAX_N) + 1) / 2 : g.m_rows);
    g.box_n = 16 * (bi + 1);
    const int blk_bytes = g.pair ? g.unit_rows * GM_BK * 2 : GM_BLK_BYTES;
    // the ring may be told to stay small enough for two CTAs (of this kernel or of the next one in
    // the stream) to share an SM, so that one's ending overlaps the other's first copies; rows
    // that do not fit such a ring take the whole SM
    auto stage_bytes = [&](int kb) { return 2 * kb * blk_bytes + 2 * kb * g.box_n * GM_BK * 2; };
    // (the exchange buffer is taken only by the ending that uses it: without it a third stage fits at up
    // to 16 rows, 123.9 -> 122.1 us a layer of the 28-layer shape at 12)
    const int xchg = Epi::XCHG && g.splits == 1 ? GM_XCHG_BYTES : 0;
    // an MMA reads 128 rows of a weight tile; where the tiles are lower, what it reads behind the last
    // one of the last stage has to be the CTA's own memory: the stage's activations, and padding
    auto pad = [&](int kb) { return std::max(0, GM_BLK_BYTES - blk_bytes - 2 * kb * g.box_n * GM_BK * 2); };
    auto plan = [&](int budget) {
        const int room = budget - 1024 - xchg - pad(1);
        // two k-blocks per copy whenever the inner dimension allows the 3-D view and two stages fit
        g.three_d = (g.K % GM_BK == 0) && !DUO && 2 * stage_bytes(2) <= room && c->tc_kb != 1;
        g.kb = g.three_d ? 2 : 1;
        g.stages = std::min(GM_MAX_STAGES, room / stage_bytes(g.kb));
        return g.stages >= 2;
    };
    if (!plan(std::min(SMEM_BUDGET, c->gemm_smem_kb * 1024)) && !plan(SMEM_BUDGET)) return cudaErrorInvalidValue;
    g.status = c->sd.counts + CNT_STATUS;
    const int n_units = g.units[0] + (g.pair ? 0 : g.units[1] + g.units[2]);
    const int k_stages = ((g.K + GM_BK - 1) / GM_BK + g.kb - 1) / g.kb;
    g.splits = std::max(1, std::min(g.splits, k_stages));
    const size_t smem = 1024 + (size_t)g.stages * stage_bytes(g.kb) + xchg + pad(g.kb);
    const int per_sm = (smem + 1024) * 2 <= 227 * 1024 ? std::max(1, c->gemm_cps) : 1;  // CTAs of this launch that fit an SM
    const int grid_x = DUO ? 2 * std::max(1, std::min(c->n_sm / 2, (n_units + 1) / 2 * g.splits))
                           : std::max(1, std::min(c->n_sm * per_sm, n_units * g.splits));
    const int grid_y = (g.m_rows + GM_MAX_N - 1) / GM_MAX_N;
    if (g.three_d)
        return launch(c, kern, dim3(grid_x, grid_y), dim3(GM_THREADS), smem, a0.m3, a1.m3, a2.m3, b_maps[bi].m3, g,
                      epi);
    return launch_clusters(c, DUO ? 2 : 1, kern, dim3(grid_x, grid_y), dim3(GM_THREADS), smem, a0.m2, a1.m2, a2.m2, b_maps[bi].m2,
                           g, epi);
}

template <class Epi>
cudaError_t launch_gemm(sparsk_ctx *c, const TmaPair &a0, const TmaPair &a1, const TmaPair &a2, const TmaPair *b_maps,
                        const GemmArgs &g, const Epi &epi)
{
    return g.m_rows <= GM_MAX_N / 2 ? launch_gemm_inst<Epi, false>(c, a0, a1, a2, b_maps, g, epi)
                                    : launch_gemm_inst<Epi, true>(c, a0, a1, a2, b_maps, g, epi);
}

cudaError_t run_norm(sparsk_ctx *c, const float *h, const bf16 *gain, const int *row_idx, int n_rows)
{
    return launch(c, rmsnorm_rows_kernel, dim3(n_rows), dim3(RN_THREADS), 0, h, gain, row_idx, c->xnorm, c->xnorm_lo, n_rows,
                  c->dm.d_model, c->dm.rms_eps);
}

// How many cuts of the inner dimension fill the machine when a product has `units` units for every block of rows.
int splits_for(const sparsk_ctx *c, int units, int m_rows)
{
    units *= div_up(m_rows, GM_MAX_N);
    const int ctas = c->n_sm * std::max(1, c->gemm_cps);
    return units * 2 <= ctas ? ctas / units : 1;
}

// One transformer layer over a row set on the tensor-core path, in two halves: the front
// (RMSNorm, q/k/v projection, rotary embedding, cache append) and the back (attention,
// O-projection, MLP).  The last layer of an upper pass runs its back half on fewer rows.
cudaError_t run_layer_tc_front(sparsk_ctx *c, int layer, float *h, const RowSet &rs)
{
    const sparsk_dims &d = c->dm;
    const int li = layer - 1, M = rs.n_rows;
    const int qd = d.n_q_heads * d.head_dim, kd = d.n_kv_heads * d.head_dim;
    const size_t lstride = (size_t)d.max_seqs * d.n_kv_heads * d.max_seq_len * d.head_dim;
    kv_t *kc = c->kcache + li * lstride, *vc = c->vcache + li * lstride;
    cudaError_t e;
    c->cur_class = KC_MISC;
    if ((e = run_norm(c, h, c->attn_norm[li], nullptr, M)) != cudaSuccess) return e;
    {
        c->cur_class = KC_QKV;
        GemmArgs g{};
        g.K = d.d_model; g.units[0] = div_up(qd, 2 * GM_BM); g.units[1] = g.units[2] = div_up(kd, 2 * GM_BM);
        g.m_rows = M;
        g.splits = splits_for(c, g.units[0] + g.units[1] + g.units[2], M);
        QkvEnd ep;
        ep.q_out = c->qbuf; ep.kc = kc; ep.vc = vc; ep.rope = c->rope;
        ep.row_slot = rs.slot; ep.row_pos = rs.pos; ep.Hq = d.n_q_heads; ep.Hkv = d.n_kv_heads; ep.hd = d.head_dim;
        ep.S = d.max_seq_len; ep.partial = g.splits > 1 ? c->qkv_part : nullptr;
        if ((e = launch_gemm(c, c->tm_wq[li], c->tm_wk[li], c->tm_wv[li], c->tm_x, g, ep)) != cudaSuccess) return e;
        if (g.splits > 1 &&
            (e = launch(c, qkv_finish_kernel, dim3(M, div_up((d.n_q_heads + 2 * d.n_kv_heads) * (d.head_dim / 2), QF_THREADS)),
                        dim3(QF_THREADS), 0, c->qkv_part, c->qbuf, kc, vc, (const float2 *)c->rope,
                        rs.slot, rs.pos, d.n_q_heads, d.n_kv_heads, d.head_dim, d.max_seq_len)) != cudaSuccess)
            return e;
    }
    c->cur_class = KC_MISC;
    return cudaSuccess;
}

cudaError_t run_layer_tc_back(sparsk_ctx *c, int layer, float *h, const RowSet &rs)
{
    const sparsk_dims &d = c->dm;
    const int li = layer - 1, M = rs.n_rows;
    const int qd = d.n_q_heads * d.head_dim;
    cudaError_t e;
    c->cur_class = KC_ATTN;
    if ((e = run_attn(c, layer, rs)) != cudaSuccess) return e;
    {
        c->cur_class = KC_OPROJ;
        GemmArgs g{};
        g.K = qd; g.units[0] = div_up(d.d_model, 2 * GM_BM); g.m_rows = M;
        g.splits = splits_for(c, g.units[0], M);
        ResidEnd ep;
        ep.h = h; ep.n_out = d.d_model; ep.atomic = 1;
        if ((e = launch_gemm(c, c->tm_wo[li], c->tm_wo[li], c->tm_wo[li], c->tm_ao, g, ep)) != cudaSuccess) return e;
    }
    c->cur_class = KC_MISC;
    if ((e = run_norm(c, h, c->mlp_norm[li], nullptr, M)) != cudaSuccess) return e;
    {
        c->cur_class = KC_GATEUP;
        GemmArgs g{};
        const int t = M > GU_EVEN_ROWS, rows = c->gu_rows[t];
        g.K = d.d_model; g.units[0] = div_up(d.d_ffn, rows); g.pair = 1; g.unit_rows = rows; g.m_rows = M; g.splits = 1;
        GateUpEnd ep;
        ep.u = c->act; ep.u_lo = c->act_lo; ep.F = d.d_ffn;
        if ((e = launch_gemm(c, c->tm_wg[t][li], c->tm_wu[t][li], c->tm_wu[t][li], c->tm_x, g, ep)) != cudaSuccess) return e;
    }
    {
        c->cur_class = KC_DOWN;
        GemmArgs g{};
        g.K = d.d_ffn; g.units[0] = div_up(d.d_model, 2 * GM_BM); g.m_rows = M;
        g.splits = splits_for(c, g.units[0], M);
        ResidEnd ep;
        ep.h = h; ep.n_out = d.d_model; ep.atomic = 1;
        e = launch_gemm(c, c->tm_wd[li], c->tm_wd[li], c->tm_wd[li], c->tm_act, g, ep);
    }
    c->cur_class = KC_MISC;
    return e;
}

bool use_tc(const sparsk_ctx *c, int n_rows) { return c->tc_ok && n_rows >= c->gemm_min_rows && c->dm.d_model >= GM_BK; }


// Head of `layer` over list `l` on the tensor-core path.
cudaError_t run_head_tc(sparsk_ctx *c, int layer, const float *h, int list, int n_rows)
{
    const sparsk_dims &d = c->dm;
    const int li = layer - 1, B = d.max_seqs, speech = list & 1;
    cudaError_t e;
    c->cur_class = KC_MISC;
    if ((e = run_norm(c, h, c->head_norm[li], c->sd.list_row + (size_t)list * B, n_rows)) != cudaSuccess) return e;
    c->cur_class = KC_HEAD;
    HeadEnd ep;
    ep.seq_of_row = c->sd.list_seq + (size_t)list * B; ep.argmax = c->sd.argmax; ep.logits = head_logits(c);
    ep.lo = speech ? d.vocab_text : 0; ep.hi = speech ? d.vocab_text + d.vocab_speech : d.vocab_text;
    ep.V = d.vocab_text + d.vocab_speech;
    GemmArgs g{};
    g.K = d.d_model; g.units[0] = div_up(ep.hi - ep.lo, 2 * GM_BM); g.row0[0] = ep.lo; g.m_rows = n_rows;
    g.splits = 1;
    e = launch_gemm(c, c->tm_head[li], c->tm_head[li], c->tm_head[li], c->tm_x, g, ep);
    c->cur_class = KC_MISC;
    return e;
}


// ---------------------------------------------------------------- persistent layer-range kernel
bool build_mega(sparsk_ctx *c)
{
    const sparsk_dims &d = c->dm;
    void *fp = nullptr;
    cudaDriverEntryPointQueryResult qr;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fp, cudaEnableDefault, &qr) != cudaSuccess || !fp ||
        qr != cudaDriverEntryPointSuccess)
        return false;
    EncodeTiledFn fn = (EncodeTiledFn)fp;
    const size_t qd = (size_t)d.n_q_heads * d.head_dim, kd = (size_t)d.n_kv_heads * d.head_dim;
    // [16 rows][256 columns] boxes of a row-major matrix, no swizzle, zero fill outside
    auto enc = [&](CUtensorMap *m, const void *base, size_t rows, size_t cols) {
        const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
        const cuuint64_t strides[1] = {(cuuint64_t)cols * 2};
        const cuuint32_t box[2] = {(cuuint32_t)MK_BOX_COLS, (cuuint32_t)MK_BOX_ROWS};
        const cuuint32_t es[2] = {1, 1};
        return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base), dims, strides, box, es,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    };
    // [64 rows][cols columns] boxes of O and down
    auto enc_col = [&](CUtensorMap *m, const void *base, size_t rows, size_t cols, int box_cols) {
        const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
        const cuuint64_t strides[1] = {(cuuint64_t)cols * 2};
        const cuuint32_t box[2] = {(cuuint32_t)box_cols, (cuuint32_t)MK_CBOX_ROWS};
        const cuuint32_t es[2] = {1, 1};
        return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base), dims, strides, box, es,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    };
    c->mk_cols16 = mk_cols(d.d_ffn, d.d_model, MK_BOX_ROWS, c->n_sm);
    c->mk_cols32 = mk_cols(d.d_ffn, d.d_model, 2 * MK_BOX_ROWS, c->n_sm);
    // The swizzled three-dimensional views need inner dimensions that are whole 64-element blocks, and
    // the RMSNorm of the form leaves whole residual rows in the activation area: 4,352 numbers.
    // Passes of three and four wider rows take the tcgen05 path.  us a layer after 1,000 positions at three / four rows, here
    // and there: 3,584 numbers (MLP 18,944) 106 / 107 and 119 / 120, 4,096 (14,336) 109 / 109 and 117 / 118, 4,352 (11,776)
    // 108 / 109 and 116 / 116, 4,352 (30,720) 179 / 180 and 189 / 189.  (Wider rows normalised a window at a time, in an earlier
    // form of this kernel: 142 / 204 at 5,120 where the tcgen05 path takes 134.)
    c->mk_tc_ok = d.d_model % 64 == 0 && d.d_ffn % 64 == 0 && qd % 64 == 0 && div_up(d.d_model, MK_BOX_COLS) <= MK_TC_STEPS;
    auto enc_sw = [&](CUtensorMap *m, const void *base, size_t rows, size_t cols) {
        const cuuint64_t dims[3] = {64, (cuuint64_t)rows, (cuuint64_t)(cols / 64)};
        const cuuint64_t strides[2] = {(cuuint64_t)cols * 2, 128};
        const cuuint32_t box[3] = {64, (cuuint32_t)MK_BOX_ROWS, (cuuint32_t)(MK_BOX_COLS / 64)};
        const cuuint32_t es[3] = {1, 1, 1};
        return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(base), dims, strides, box, es,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    };
    auto enc_col_sw = [&](CUtensorMap *m, const void *base, size_t rows, size_t cols, int box_cols) {
        const cuuint64_t dims[3] = {32, (cuuint64_t)rows, (cuuint64_t)(cols / 32)};
        const cuuint64_t strides[2] = {(cuuint64_t)cols * 2, 64};
        const cuuint32_t box[3] = {32, (cuuint32_t)MK_CBOX_ROWS, (cuuint32_t)(box_cols / 32)};
        const cuuint32_t es[3] = {1, 1, 1};
        return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(base), dims, strides, box, es,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    };
    c->mk_host.resize(d.n_layers);
    bool ok = true;
    for (int l = 0; l < d.n_layers; l++) {
        MkLayer &m = c->mk_host[l];
        memset(&m, 0, sizeof m);
        const void *mats[MKW_N] = {c->wq[l], c->wk[l], c->wv[l], c->wo[l], c->w_gate[l], c->w_up[l], c->w_down[l]};
        const size_t rows[MKW_N] = {qd, kd, kd, (size_t)d.d_model, (size_t)d.d_ffn, (size_t)d.d_ffn, (size_t)d.d_model};
        const size_t cols[MKW_N] = {(size_t)d.d_model, (size_t)d.d_model, (size_t)d.d_model, qd, (size_t)d.d_model,
                                    (size_t)d.d_model, (size_t)d.d_ffn};
        for (int k = 0; k < MKW_N; k++) {
            if (k == MKW_O || k == MKW_D) {
                ok = ok && enc_col(&m.map[k], mats[k], rows[k], cols[k], k == MKW_O ? d.head_dim : c->mk_cols16.box);
                if (c->mk_tc_ok) ok = ok && enc_col_sw(&m.map[MKW_N + k], mats[k], rows[k], cols[k], k == MKW_O ? d.head_dim : c->mk_cols32.box);
            } else {
                ok = ok && enc(&m.map[k], mats[k], rows[k], cols[k]);
                if (c->mk_tc_ok) ok = ok && enc_sw(&m.map[MKW_N + k], mats[k], rows[k], cols[k]);
            }
        }
        if (c->attn_tma_ok) {
            m.kmap = c->tm_kc16[l];
            m.vmap = c->tm_vc16[l];
        }
        m.attn_gain = c->attn_norm[l];
        m.mlp_gain = c->mlp_norm[l];
    }
    if (!ok) return false;
    if (cudaMemcpyAsync(c->mk_layers, c->mk_host.data(), sizeof(MkLayer) * d.n_layers, cudaMemcpyHostToDevice,
                        c->stream) != cudaSuccess ||
        cudaMemsetAsync(c->mk_bar, 0, sizeof(unsigned long long), c->stream) != cudaSuccess ||
        cudaMemsetAsync(c->mk_abort, 0, sizeof(int), c->stream) != cudaSuccess ||
        cudaMemsetAsync(c->mk_h2, 0, sizeof(float) * MK_MAX_ROWS * (size_t)d.d_model, c->stream) != cudaSuccess)
        return false;
    c->mk_bar_base = 0;
    int dev = 0, coop = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess)
        return false;
    c->mk_coop = coop;
    return true;
}

// Can a pass of n_rows rows go through the persistent kernel?
bool use_mega(const sparsk_ctx *c, int n_rows)
{
    return c->mega && c->mk_ok && c->mk_coop && n_rows >= 1 && n_rows <= c->mk_max_rows && (n_rows < MK_TC_ROWS || c->mk_tc_ok) &&
           c->attn_tma_ok && c->n_sm <= MK_MAX_CTAS &&
           (size_t)MK_MAX_ROWS * c->dm.n_kv_heads * (c->dm.max_seq_len / AT_TP + 1) * MK_MAX_CTAS < (1ull << 31);  // (32-bit shares)
}

template <int M, int HD, bool WIDE>
cudaError_t launch_mega_form(sparsk_ctx *c, const MkArgs &a)
{
    constexpr size_t smem = mk_smem_bytes(M, WIDE);
    static PerDevice<int> grid_dev;  // 0: not asked yet, 1: one CTA per SM fits, 2: it does not
    int &grid_ok = grid_dev.here();
    auto kern = mega_kernel<M, HD, WIDE>;
    if (grid_ok == 0) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        int per_sm = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, MK_THREADS, smem);
        if (e != cudaSuccess) return e;
        grid_ok = per_sm >= 1 ? 1 : 2;
    }
    if (grid_ok != 1) return cudaErrorCooperativeLaunchTooLarge;
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof cfg);
    cfg.gridDim = dim3(c->n_sm);
    cfg.blockDim = dim3(MK_THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = c->stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    c->launches++;
    const bool timed = (c->time_class == KC_MEGA || c->time_class == KC_ALL) && c->tev_used + 2 <= c->tev.size();
    if (timed) {
        c->tev_class[c->tev_used / 2] = KC_MEGA;
        cudaEventRecord(c->tev[c->tev_used++], c->stream);
    }
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, a);
    if (timed) cudaEventRecord(c->tev[c->tev_used++], c->stream);
    return e;
}

template <int M, int HD>
cudaError_t launch_mega_inst(sparsk_ctx *c, const MkArgs &a)
{
    return a.cols.wide ? launch_mega_form<M, HD, true>(c, a) : launch_mega_form<M, HD, false>(c, a);
}

// Layers [l_begin, l_end) (0-based) over a row set of one to four rows, in one launch.
cudaError_t run_mega(sparsk_ctx *c, int l_begin, int l_end, float *h, const RowSet &rs)
{
    const sparsk_dims &d = c->dm;
    MkArgs a{};
    a.layers = c->mk_layers; a.layer_begin = l_begin; a.layer_end = l_end; a.h = h;
    a.row_slot = rs.slot; a.row_pos = rs.pos; a.grp_row0 = rs.grp_row0; a.grp_nrows = rs.grp_nrows;
    a.n_rows = rs.n_rows; a.n_groups = rs.n_groups_h;
    a.h2 = c->mk_h2;
    a.act = c->mk_act;
    a.kc = c->kcache; a.vc = c->vcache;
    a.kv_layer = (size_t)d.max_seqs * d.n_kv_heads * d.max_seq_len * d.head_dim;
    a.q_buf = c->qbuf; a.part_o = c->part_o; a.part_ml = c->part_ml;
    a.rope = c->rope;
    a.d = d.d_model; a.Hq = d.n_q_heads; a.Hkv = d.n_kv_heads; a.hd = d.head_dim; a.F = d.d_ffn; a.S = d.max_seq_len;
    a.n_slots = d.max_seqs; a.eps = d.rms_eps;
    a.cols = rs.n_rows >= MK_TC_ROWS ? c->mk_cols32 : c->mk_cols16;
    a.bar = c->mk_bar; a.bar_base = c->mk_bar_base; a.abort_word = c->mk_abort; a.status = c->sd.counts + CNT_STATUS;
    if (c->inject_timeout) {
        // the launch is told a barrier count that is never reached: its first grid barrier runs
        // into the wall-clock limit, every CTA gives up and the step reports SPARSK_ETIMEOUT
        a.bar_base += 1ull << 40;
        c->inject_timeout = 0;
    }
    a.short_copy_layer = -1;
    if (c->inject_short_copy && l_end - l_begin >= 2) {
        a.short_copy_layer = l_begin + 1;
        c->inject_short_copy = 0;
    }
    a.trace = c->mk_trace;
    c->mk_trace_n = 1 + mk_phases(a.cols.wide) * (l_end - l_begin);
    c->mk_bar_base += (unsigned long long)mk_phases(a.cols.wide) * (unsigned long long)(l_end - l_begin) * (unsigned long long)c->n_sm;
    // (three rows run as four with one masked)
    if (d.head_dim == 128) {
        switch (rs.n_rows) {
        case 1: return launch_mega_inst<1, 128>(c, a);
        case 2: return launch_mega_inst<2, 128>(c, a);
        default: return launch_mega_inst<4, 128>(c, a);
        }
    }
    switch (rs.n_rows) {
    case 1: return launch_mega_inst<1, 64>(c, a);
    case 2: return launch_mega_inst<2, 64>(c, a);
    default: return launch_mega_inst<4, 64>(c, a);
    }
}

// Front half of a layer over a row set: q to the query buffer, k and v into the cache.
cudaError_t run_layer_front(sparsk_ctx *c, int layer, float *h, const RowSet &rs)
{
    if (use_tc(c, rs.n_rows)) return run_layer_tc_front(c, layer, h, rs);
    c->cur_class = KC_QKV;
    const cudaError_t e = run_qkv(c, layer, h, rs);
    c->cur_class = KC_MISC;
    return e;
}

// Back half: attention, O-projection and MLP; h <- h^(layer).
cudaError_t run_layer_back(sparsk_ctx *c, int layer, float *h, const RowSet &rs)
{
    const sparsk_dims &d = c->dm;
    const int li = layer - 1;
    cudaError_t e;
    if (use_tc(c, rs.n_rows)) return run_layer_tc_back(c, layer, h, rs);
    c->cur_class = KC_ATTN;
    if ((e = run_attn(c, layer, rs)) != cudaSuccess) return e;
    c->cur_class = KC_OPROJ;
    if ((e = run_resid(c, c->wo[li], c->attn_o, h, d.n_q_heads * d.head_dim, d.d_model, rs.n_rows)) != cudaSuccess) return e;
    c->cur_class = KC_GATEUP;
    if ((e = run_gateup(c, layer, h, rs.n_rows)) != cudaSuccess) return e;
    c->cur_class = KC_DOWN;
    e = run_resid(c, c->w_down[li], c->act, h, d.d_ffn, d.d_model, rs.n_rows);
    c->cur_class = KC_MISC;
    return e;
}

// One transformer layer over a row set: h <- h^(layer).
cudaError_t run_layer(sparsk_ctx *c, int layer, float *h, const RowSet &rs)
{
    const cudaError_t e = run_layer_front(c, layer, h, rs);
    return e != cudaSuccess ? e : run_layer_back(c, layer, h, rs);
}

// Layers l_first..l_last (1-based, inclusive) over a row set.
cudaError_t run_layers(sparsk_ctx *c, int l_first, int l_last, float *h, const RowSet &rs)
{
    if (l_first > l_last) return cudaSuccess;
    const int n_layers = l_last - l_first + 1;
    if (use_mega(c, rs.n_rows)) {
        c->route_layers[0] += n_layers;
        return run_mega(c, l_first - 1, l_last, h, rs);
    }
    c->route_layers[use_tc(c, rs.n_rows) ? 1 : 2] += n_layers;
    for (int l = l_first; l <= l_last; l++) {
        const cudaError_t e = run_layer(c, l, h, rs);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

bool good(const sparsk_ctx *c) { return c && c->magic == CTX_MAGIC; }

}  // namespace

// =============================================================================== C ABI

extern "C" size_t sparsk_workspace_bytes(const sparsk_dims *dims)
{
    if (!dims_ok(dims)) return 0;
    return carve(nullptr, dims, nullptr);
}

extern "C" int sparsk_create(const sparsk_dims *dims, const sparsk_weights *w, void *workspace,
                             size_t workspace_bytes, void *cuda_stream, sparsk_ctx **out)
{
    if (!out) return SPARSK_EINVAL;
    *out = nullptr;
    if (!dims_ok(dims) || !w || !workspace) return SPARSK_EINVAL;
    if ((uintptr_t)workspace % 256) return SPARSK_EINVAL;
    if (workspace_bytes < sparsk_workspace_bytes(dims)) return SPARSK_EINVAL;
    const int L = dims->n_layers, e = dims->exit_layer;
    const void *const *arrs[] = {w->attn_norm, w->wq, w->wk, w->wv, w->wo, w->mlp_norm, w->w_gate, w->w_up, w->w_down};
    if (!w->embed || ((uintptr_t)w->embed % 16) || !w->head_norm || !w->head_proj) return SPARSK_EINVAL;
    for (auto a : arrs) {
        if (!a) return SPARSK_EINVAL;
        for (int l = 0; l < L; l++)
            if (!a[l] || ((uintptr_t)a[l] % 16)) return SPARSK_EINVAL;
    }
    for (int l = 0; l < L; l++)
        if (((uintptr_t)w->head_norm[l] % 16) || ((uintptr_t)w->head_proj[l] % 16)) return SPARSK_EINVAL;
    if (((size_t)dims->vocab_text * dims->d_model * 2) % 16) return SPARSK_EINVAL;
    // the heads of layers e and L are what the periodic schedule reads
    if (!w->head_norm[L - 1] || !w->head_proj[L - 1]) return SPARSK_ENOHEAD;
    if (dims->refresh_period > 1 && e < L && (!w->head_norm[e - 1] || !w->head_proj[e - 1])) return SPARSK_ENOHEAD;
    if (dims->conf_modalities)   // the confidence rule consults the head of every layer from conf_start on
        for (int l = dims->conf_start; l < L; l++)
            if (!w->head_norm[l - 1] || !w->head_proj[l - 1]) return SPARSK_ENOHEAD;

    sparsk_ctx *ctx = new (std::nothrow) sparsk_ctx();
    if (!ctx) return SPARSK_EINVAL;
    ctx->magic = CTX_MAGIC;
    ctx->dm = *dims;
    ctx->dm.prefill_rows = prefill_rows_of(dims);
    ctx->stream = (cudaStream_t)cuda_stream;
    ctx->err[0] = 0;
    auto cp = [&](std::vector<const bf16 *> &dst, const void *const *src) {
        dst.resize(L);
        for (int l = 0; l < L; l++) dst[l] = (const bf16 *)src[l];
    };
    cp(ctx->attn_norm, w->attn_norm); cp(ctx->wq, w->wq); cp(ctx->wk, w->wk); cp(ctx->wv, w->wv);
    cp(ctx->wo, w->wo); cp(ctx->mlp_norm, w->mlp_norm); cp(ctx->w_gate, w->w_gate); cp(ctx->w_up, w->w_up);
    cp(ctx->w_down, w->w_down); cp(ctx->head_norm, w->head_norm); cp(ctx->head_proj, w->head_proj);
    ctx->embed = (const bf16 *)w->embed;
    ctx->cap_rows = cap_rows_of(&ctx->dm);
    carve(ctx, &ctx->dm, (char *)workspace);
    ctx->h_len.assign(dims->max_seqs, 0);
    ctx->h_pend.assign(dims->max_seqs, 0);
    ctx->pdl = 1; ctx->attn_split = 0; ctx->gemm_min_rows = 3;
    ctx->tc_ok = false;
    ctx->tc_kb = 0;
    ctx->gemm_smem_kb = 220;
    ctx->gemm_cps = 1;
    ctx->mk_max_rows = MK_MAX_ROWS;
    ctx->attn_tc = 1; ctx->attn_tc_min_q = 33; ctx->attn_stages = AW_NST;
    ctx->inject_timeout = ctx->inject_short_copy = 0;
    ctx->attn_ticket_base = 0; ctx->attn_dynamic = 1; ctx->attn_ctas = 0;
    ctx->attn_tma = 1; ctx->attn_tma_ok = 0;
    ctx->trim_last = 1;
    ctx->conf_host = nullptr; ctx->conf_ent_host = nullptr;
    ctx->h_fill.assign(dims->max_seqs, std::vector<int>());
    for (auto &v : ctx->route_layers) v = 0;
    ctx->mega = 1; ctx->mk_ok = 0; ctx->mk_coop = 0; ctx->mk_bar_base = 0; ctx->mk_trace_n = 0;
    ctx->gv_ks = 0; ctx->gv_r = 0;
    ctx->dbg_hidden = nullptr; ctx->dbg_logits = nullptr;
    ctx->samp_temperature = 0.f; ctx->samp_top_p = 1.f; ctx->samp_uniforms = nullptr; ctx->samp_scratch = nullptr;
    ctx->launches = 0;
    ctx->cur_class = KC_MISC; ctx->time_class = KC_MISC; ctx->tev_used = 0;
    ctx->stage_next = 0;
    for (int i = 0; i < STAGE_RING; i++) { ctx->stage_host[i] = nullptr; ctx->stage_ev[i] = nullptr; }
    ctx->io_host = nullptr;

    int rc = SPARSK_OK;
    do {
        int dev = 0;
        cudaError_t ce;
        if ((ce = cudaGetDevice(&dev)) != cudaSuccess ||
            (ce = cudaDeviceGetAttribute(&ctx->n_sm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) {
            rc = fail(ctx, SPARSK_ECUDA, "device query failed: %s", cudaGetErrorString(ce));
            break;
        }
        for (int i = 0; i < STAGE_RING && rc == SPARSK_OK; i++) {
            if ((ce = cudaHostAlloc((void **)&ctx->stage_host[i], 3 * sizeof(int) * dims->max_seqs, cudaHostAllocDefault)) != cudaSuccess ||
                (ce = cudaEventCreateWithFlags(&ctx->stage_ev[i], cudaEventDisableTiming)) != cudaSuccess)
                rc = fail(ctx, SPARSK_ECUDA, "staging setup failed: %s", cudaGetErrorString(ce));
        }
        if (rc == SPARSK_OK &&
            (ce = cudaHostAlloc((void **)&ctx->io_host, sizeof(int) * (3 * (size_t)dims->max_seqs + 1), cudaHostAllocDefault)) != cudaSuccess)
            rc = fail(ctx, SPARSK_ECUDA, "staging setup failed: %s", cudaGetErrorString(ce));
        if (rc) break;
        if (dims->conf_modalities) {
            // one region per segment of a step (at most one per layer, plus lists per consulted layer)
            ctx->conf_seg_ints = 4 * (size_t)ctx->cap_rows + 4 * (size_t)dims->max_seqs + 8;
            ctx->conf_host_ints = ctx->conf_seg_ints * (2 * (size_t)L + 4);
            if ((ce = cudaHostAlloc((void **)&ctx->conf_host, ctx->conf_host_ints * sizeof(int), cudaHostAllocDefault)) != cudaSuccess ||
                (ce = cudaHostAlloc((void **)&ctx->conf_ent_host, sizeof(float) * dims->max_seqs, cudaHostAllocDefault)) != cudaSuccess) {
                rc = fail(ctx, SPARSK_ECUDA, "staging setup failed: %s", cudaGetErrorString(ce));
                break;
            }
        }
        // no silent change of path: without TMA descriptors the batched path cannot run
        ctx->tc_ok = build_maps(ctx);
        if (!ctx->tc_ok) {
            rc = fail(ctx, SPARSK_ECUDA, "building the TMA descriptors failed");
            break;
        }
        ctx->mk_ok = build_mega(ctx) ? 1 : 0;
        if (!ctx->mk_ok) {
            rc = fail(ctx, SPARSK_ECUDA, "setting up the persistent layer kernel failed");
            break;
        }
        // rotary table in double, stored as float (cos, sin)
        const int half = dims->head_dim / 2;
        std::vector<float2> tab((size_t)dims->max_seq_len * half);
        for (int i = 0; i < half; i++) {
            const double inv = std::pow((double)dims->rope_base, -2.0 * i / dims->head_dim);
            for (int p = 0; p < dims->max_seq_len; p++) {
                const double th = (double)p * inv;
                tab[(size_t)p * half + i] = make_float2((float)std::cos(th), (float)std::sin(th));
            }
        }
        if ((ce = cudaMemcpyAsync(ctx->rope, tab.data(), tab.size() * sizeof(float2), cudaMemcpyHostToDevice, ctx->stream)) != cudaSuccess ||
            // the cache starts out as zeros: the tcgen05 attention kernel multiplies whole 64-position
            // tiles, and a masked weight of zero times an unwritten NaN pattern would still be NaN
            (ce = cudaMemsetAsync(ctx->kcache, 0, sizeof(kv_t) * (size_t)dims->n_layers * dims->max_seqs * dims->n_kv_heads * dims->max_seq_len * dims->head_dim, ctx->stream)) != cudaSuccess ||
            (ce = cudaMemsetAsync(ctx->vcache, 0, sizeof(kv_t) * (size_t)dims->n_layers * dims->max_seqs * dims->n_kv_heads * dims->max_seq_len * dims->head_dim, ctx->stream)) != cudaSuccess ||
            (ce = cudaMemsetAsync(ctx->kv_len, 0, sizeof(int) * dims->max_seqs, ctx->stream)) != cudaSuccess ||
            (ce = cudaMemsetAsync(ctx->pend_cnt, 0, sizeof(int) * dims->max_seqs, ctx->stream)) != cudaSuccess ||
            (ce = cudaMemsetAsync(ctx->sd.counts, 0, sizeof(int) * 8, ctx->stream)) != cudaSuccess ||
            (ce = cudaMemsetAsync(ctx->attn_ticket, 0, sizeof(unsigned), ctx->stream)) != cudaSuccess ||
            (ce = cudaMemsetAsync(ctx->qkv_part, 0, sizeof(float) * (size_t)ctx->cap_rows * (dims->n_q_heads + 2 * dims->n_kv_heads) * dims->head_dim, ctx->stream)) != cudaSuccess ||
            (ce = cudaStreamSynchronize(ctx->stream)) != cudaSuccess) {
            rc = fail(ctx, SPARSK_ECUDA, "table upload failed: %s", cudaGetErrorString(ce));
            break;
        }
    } while (0);
    if (rc != SPARSK_OK) {
        sparsk_destroy(ctx);
        return rc;
    }
    *out = ctx;
    return SPARSK_OK;
}

extern "C" int sparsk_destroy(sparsk_ctx *ctx)
{
    if (!good(ctx)) return SPARSK_ESTATE;
    cudaStreamSynchronize(ctx->stream);
    for (int i = 0; i < STAGE_RING; i++) {
        if (ctx->stage_host[i]) cudaFreeHost(ctx->stage_host[i]);
        if (ctx->stage_ev[i]) cudaEventDestroy(ctx->stage_ev[i]);
    }
    if (ctx->io_host) cudaFreeHost(ctx->io_host);
    for (cudaEvent_t ev : ctx->tev) cudaEventDestroy(ev);
    if (ctx->conf_host) cudaFreeHost(ctx->conf_host);
    if (ctx->conf_ent_host) cudaFreeHost(ctx->conf_ent_host);
    ctx->magic = 0;
    delete ctx;
    return SPARSK_OK;
}

extern "C" const char *sparsk_last_error(const sparsk_ctx *ctx) { return good(ctx) ? ctx->err : "invalid context"; }
extern "C" int64_t sparsk_launch_count(const sparsk_ctx *ctx) { return good(ctx) ? ctx->launches : -1; }
extern "C" int sparsk_conf_entropies(const sparsk_ctx *ctx, int32_t n_seqs, float *out)
{
    if (!good(ctx)) return SPARSK_ESTATE;
    const int L = ctx->dm.n_layers;
    if (!out || n_seqs < 0 || (size_t)n_seqs * L > ctx->conf_trace.size()) return SPARSK_EINVAL;
    for (size_t k = 0; k < (size_t)n_seqs * L; k++) out[k] = ctx->conf_trace[k];
    return SPARSK_OK;
}
extern "C" int sparsk_route_counts(const sparsk_ctx *ctx, int64_t *layer_passes)
{
    if (!good(ctx)) return SPARSK_ESTATE;
    if (!layer_passes) return SPARSK_EINVAL;
    for (int i = 0; i < 3; i++) layer_passes[i] = ctx->route_layers[i];
    return SPARSK_OK;
}

extern "C" int sparsk_set_debug(sparsk_ctx *ctx, float *exit_hidden, float *exit_logits)
{
    if (!good(ctx)) return SPARSK_ESTATE;
    ctx->dbg_hidden = exit_hidden;
    ctx->dbg_logits = exit_logits;
    return SPARSK_OK;
}

extern "C" size_t sparsk_sampling_scratch_bytes(const sparsk_dims *dims)
{
    if (!dims_ok(dims)) return 0;
    return (size_t)dims->max_seqs * ((size_t)dims->vocab_text + dims->vocab_speech) * sizeof(float);
}

extern "C" int sparsk_set_sampling(sparsk_ctx *ctx, float temperature, float top_p, const float *uniforms, void *scratch,
                                   size_t scratch_bytes)
{
    if (!good(ctx)) return SPARSK_ESTATE;
    if (!uniforms) {  // back to greedy decoding
        ctx->samp_uniforms = nullptr;
        ctx->samp_scratch = nullptr;
        return SPARSK_OK;
    }
    if (ctx->dm.conf_modalities)
        return fail(ctx, SPARSK_EINVAL, "set_sampling: a context with confidence-based exit decodes greedily");
    if (!(temperature > 0.f) || !(temperature < INFINITY) || !(top_p > 0.f) || !(top_p <= 1.f))
        return fail(ctx, SPARSK_EINVAL, "set_sampling: temperature %g, top_p %g", (double)temperature, (double)top_p);
    if (ctx->dm.vocab_text > SP_MAX_RANGE || ctx->dm.vocab_speech > SP_MAX_RANGE)
        return fail(ctx, SPARSK_ECAPACITY, "set_sampling: a modality has more than %d ids", SP_MAX_RANGE);
    if (!scratch || ((uintptr_t)scratch % 16) || scratch_bytes < sparsk_sampling_scratch_bytes(&ctx->dm))
        return fail(ctx, SPARSK_EINVAL, "set_sampling: scratch of %zu bytes, need %zu (16-byte aligned)", scratch_bytes,
                    sparsk_sampling_scratch_bytes(&ctx->dm));
    ctx->samp_temperature = temperature;
    ctx->samp_top_p = top_p;
    ctx->samp_uniforms = uniforms;
    ctx->samp_scratch = (float *)scratch;
    return SPARSK_OK;
}

extern "C" int sparsk_set_option(sparsk_ctx *ctx, const char *name, int64_t value)
{
    if (!good(ctx)) return SPARSK_ESTATE;
    if (!name) return fail(ctx, SPARSK_EINVAL, "option name is NULL");
    if (!strcmp(name, "gemm_min_rows") && value >= 1) ctx->gemm_min_rows = (int)std::min<int64_t>(value, 1 << 30);
    else if (!strcmp(name, "pdl") && (value == 0 || value == 1)) ctx->pdl = (int)value;
    else if (!strcmp(name, "attn_split") && value >= 0 && value <= (1 << 24)) ctx->attn_split = (int)value;
    else if (!strcmp(name, "gemv_ks") && (value == 0 || value == 1 || value == 2 || value == 4 || value == 8 || value == 16)) ctx->gv_ks = (int)value;
    else if (!strcmp(name, "mega") && (value == 0 || value == 1)) ctx->mega = (int)value;
    else if (!strcmp(name, "attn_stages") && (value == 2 || value == 3)) ctx->attn_stages = (int)value;
    else if (!strcmp(name, "attn_dynamic") && (value == 0 || value == 1)) ctx->attn_dynamic = (int)value;
    else if (!strcmp(name, "attn_tma") && (value == 0 || value == 1)) ctx->attn_tma = (int)value;
    else if (!strcmp(name, "attn_ctas") && value >= 0 && value <= 65535) ctx->attn_ctas = (int)value;
    else if (!strcmp(name, "attn_tc") && (value == 0 || value == 1)) ctx->attn_tc = (int)value;
    else if (!strcmp(name, "attn_tc_min_q") && value >= 1 && value <= (1 << 20)) ctx->attn_tc_min_q = (int)value;
    else if (!strcmp(name, "mega_max_rows") && value >= 1 && value <= MK_MAX_ROWS) ctx->mk_max_rows = (int)value;
    else if (!strcmp(name, "gemm_kb") && (value == 0 || value == 1)) ctx->tc_kb = (int)value;
    else if (!strcmp(name, "gemm_ctas_per_sm") && (value == 1 || value == 2)) ctx->gemm_cps = (int)value;
    else if (!strcmp(name, "gemm_smem_kb") && value >= 48 && value <= 220) ctx->gemm_smem_kb = (int)value;
    else if (!strcmp(name, "trim_last_layer") && value >= 0 && value <= 2) ctx->trim_last = (int)value;
    else if (!strcmp(name, "inject_barrier_timeout") && (value == 0 || value == 1)) ctx->inject_timeout = (int)value;
    else if (!strcmp(name, "inject_short_copy") && (value == 0 || value == 1)) ctx->inject_short_copy = (int)value;
    else if (!strcmp(name, "gemv_r") && (value == 0 || value == 1 || value == 2 || value == 4)) ctx->gv_r = (int)value;
    else if (!strcmp(name, "time_kernel") && value >= 0 && value <= KC_ALL) {
        // start (or stop, with 0) timing every launch of one kernel class; resets the totals
        if (value && ctx->tev.empty()) {
            ctx->tev.resize(2 * TIME_POOL);
            ctx->tev_class.assign(TIME_POOL, 0);
            for (auto &ev : ctx->tev) CU(cudaEventCreate(&ev));
        }
        ctx->time_class = (int)value;
        ctx->tev_used = 0;
    } else return fail(ctx, SPARSK_EINVAL, "unknown option or bad value: %s=%lld", name, (long long)value);
    return SPARSK_OK;
}

extern "C" int sparsk_kernel_time(sparsk_ctx *ctx, double *total_ms, int64_t *n_launches)
{
    if (!good(ctx)) return SPARSK_ESTATE;
    if (!total_ms || !n_launches) return fail(ctx, SPARSK_EINVAL, "kernel_time: NULL output");
    CU(cudaStreamSynchronize(ctx->stream));
    double tot = 0.0;
    for (size_t i = 0; i + 1 < ctx->tev_used; i += 2) {
        float ms = 0.f;
        CU(cudaEventElapsedTime(&ms, ctx->tev[i], ctx->tev[i + 1]));
        tot += ms;
    }
    *total_ms = tot;
    *n_launches = (int64_t)(ctx->tev_used / 2);
    return SPARSK_OK;
}

// Reads and clears the device status word (the stream is synchronised) and turns it into a
// return code.  After a timeout the persistent kernels' grid-barrier counter, its host mirror and
// the abort word start over, so that the next launch does not find a stale abort request or a
// counter that no longer matches its base.
static int act_on_status(sparsk_ctx *ctx, int status);
static int read_status(sparsk_ctx *ctx)
{
    int status = 0;
    CU(cudaMemcpyAsync(&status, ctx->sd.counts + CNT_STATUS, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
    CU(cudaStreamSynchronize(ctx->stream));
    return act_on_status(ctx, status);
}
// What a status word read back from the device (the stream is idle) means for the caller.
static int act_on_status(sparsk_ctx *ctx, int status)
{
    if (status) CU(cudaMemsetAsync(ctx->sd.counts + CNT_STATUS, 0, sizeof(int), ctx->stream));
    if (status & ST_TIMEOUT) {
        CU(cudaMemsetAsync(ctx->mk_bar, 0, sizeof(unsigned long long), ctx->stream));
        CU(cudaMemsetAsync(ctx->mk_abort, 0, sizeof(int), ctx->stream));
        CU(cudaMemsetAsync(ctx->mk_h2, 0, sizeof(float) * MK_MAX_ROWS * (size_t)ctx->dm.d_model, ctx->stream));
        CU(cudaMemsetAsync(ctx->attn_ticket, 0, sizeof(unsigned), ctx->stream));
        ctx->mk_bar_base = 0;
        ctx->attn_ticket_base = 0;
        return fail(ctx, SPARSK_ETIMEOUT, "a bounded in-kernel wait ran out");
    }
    if (status & ST_BAD_TOKEN) return fail(ctx, SPARSK_EINVAL, "a token id was outside the vocabulary (clamped)");
    return SPARSK_OK;
}

extern "C" int sparsk_check(sparsk_ctx *ctx)
{
    if (!good(ctx)) return SPARSK_ESTATE;
    return read_status(ctx);
}

extern "C" int sparsk_kernel_time_by_class(sparsk_ctx *ctx, double *total_ms, int64_t *n_launches)
{
    if (!good(ctx)) return SPARSK_ESTATE;
    if (!total_ms || !n_launches) return fail(ctx, SPARSK_EINVAL, "kernel_time_by_class: NULL output");
    CU(cudaStreamSynchronize(ctx->stream));
    for (int k = 0; k < 8; k++) {
        total_ms[k] = 0.0;
        n_launches[k] = 0;
    }
    for (size_t i = 0; i + 1 < ctx->tev_used; i += 2) {
        float ms = 0.f;
        CU(cudaEventElapsedTime(&ms, ctx->tev[i], ctx->tev[i + 1]));
        const int k = ctx->tev_class[i / 2] & 7;
        total_ms[k] += ms;
        n_launches[k]++;
    }
    return SPARSK_OK;
}

extern "C" int sparsk_phase_trace(sparsk_ctx *ctx, int64_t *out_ns, int32_t capacity)
{
    if (!good(ctx)) return SPARSK_ESTATE;
    if (!out_ns || capacity < 0) return fail(ctx, SPARSK_EINVAL, "phase_trace: bad arguments");
    const int n = std::min<int>(capacity, ctx->mk_trace_n);
    if (n > 0) CU(cudaMemcpyAsync(out_ns, ctx->mk_trace, sizeof(int64_t) * n, cudaMemcpyDeviceToHost, ctx->stream));
    CU(cudaStreamSynchronize(ctx->stream));
    return n;
}

extern "C" int sparsk_reset_slot(sparsk_ctx *ctx, int32_t slot) { return sparsk_set_len(ctx, slot, 0); }

extern "C" int sparsk_set_len(sparsk_ctx *ctx, int32_t slot, int32_t len)
{
    if (!good(ctx)) return SPARSK_ESTATE;
    if (slot < 0 || slot >= ctx->dm.max_seqs || len < 0 || len > ctx->dm.max_seq_len)
        return fail(ctx, SPARSK_EINVAL, "set_len: slot %d / len %d out of range", slot, len);
    CU(launch(ctx, set_int_kernel, dim3(1), dim3(1), 0, ctx->kv_len + slot, (int)len));
    CU(launch(ctx, set_int_kernel, dim3(1), dim3(1), 0, ctx->pend_cnt + slot, 0));
    ctx->h_len[slot] = len;
    ctx->h_pend[slot] = 0;
    ctx->h_fill[slot].clear();
    return SPARSK_OK;
}

extern "C" int sparsk_slot_state(const sparsk_ctx *ctx, int32_t slot, int32_t *len, int32_t *pending)
{
    if (!good(ctx)) return SPARSK_ESTATE;
    if (slot < 0 || slot >= ctx->dm.max_seqs) return SPARSK_EINVAL;
    if (len) *len = ctx->h_len[slot];
    if (pending) *pending = ctx->h_pend[slot];
    return SPARSK_OK;
}

static int kv_io(sparsk_ctx *ctx, int32_t slot, int32_t layer, int32_t first_pos, int32_t n, void *k, void *v, int to_cache)
{
    if (!good(ctx)) return SPARSK_ESTATE;
    const sparsk_dims &d = ctx->dm;
    if (slot < 0 || slot >= d.max_seqs || layer < 1 || layer > d.n_layers || first_pos < 0 || n < 0 ||
        (long)first_pos + n > d.max_seq_len || !k || !v)
        return fail(ctx, SPARSK_EINVAL, "kv import/export: argument out of range");
    if (n == 0) return SPARSK_OK;
    const size_t per_slot = (size_t)d.n_kv_heads * d.max_seq_len * d.head_dim;
    const size_t off = ((size_t)(layer - 1) * d.max_seqs + slot) * per_slot;
    const size_t total = (size_t)n * d.n_kv_heads * d.head_dim;
    const int blocks = (int)std::min<size_t>((total + 255) / 256, 4096);
    CU(launch(ctx, kv_copy_kernel, dim3(blocks), dim3(256), 0, ctx->kcache + off, ctx->vcache + off, (kv_t *)k,
              (kv_t *)v, (int)first_pos, (int)n, d.n_kv_heads, d.head_dim, d.max_seq_len, to_cache));
    return SPARSK_OK;
}
extern "C" int sparsk_import_kv(sparsk_ctx *ctx, int32_t slot, int32_t layer, int32_t first_pos, int32_t n,
                                const void *k, const void *v)
{
    return kv_io(ctx, slot, layer, first_pos, n, const_cast<void *>(k), const_cast<void *>(v), 1);
}
extern "C" int sparsk_export_kv(sparsk_ctx *ctx, int32_t slot, int32_t layer, int32_t first_pos, int32_t n,
                                void *k, void *v)
{
    return kv_io(ctx, slot, layer, first_pos, n, k, v, 0);
}

// --------------------------------------------------------------------------- prefill
// Rows of the next pass when `left` prompt rows are to come and a pass takes up to `chunk`.  A block of few rows behind whole
// ones costs a launch as much as a whole block, if its units need another wave: it is left for the next pass then, whose own launches
// cut the inner dimension or go through the persistent kernel.  us a layer in one pass / in two: 257 rows 359 / 319, 288
// rows 384 / 356, 320 rows 396 / 380, 400 rows 399 / 454 (28-layer shape; 40-layer shape 372 / 318, 374 / 347, 388 / 376, 394 / 442).
// More than 32 rows do so only if their block fills two fifths of a wave and more (those two shapes all of one and 34 of 74 pairs
// of SMs; d_ffn 8,192 at three blocks 22: 517 rows 254 / 262); where the block finds idle SMs (d_ffn 8,192 at two) 257 rows take 168 / 194.
constexpr int PREFILL_TAIL = 32;
static int prefill_pass_rows(const sparsk_ctx *c, long left, int chunk)
{
    const int n = (int)std::min<long>(chunk, left), blocks = n / GM_MAX_N, tail = n % GM_MAX_N;
    if (blocks == 0) return n;
    const int pairs = std::max(1, c->n_sm / 2), units = div_up(c->dm.d_ffn, 2 * GM_BM);  // of gate/up, a block of rows
    // those of the last block for which the waves of the blocks before it have no room
    const int beyond = units * (blocks + 1) - div_up(units * blocks, pairs) * pairs;
    return beyond > 0 && tail <= (beyond * 5 >= pairs * 2 ? 2 : 1) * PREFILL_TAIL ? n - tail : n;
}

// Few rows behind a long prefix beside a prompt's many rows: the partials have room for fewer splits the more rows a pass has
// (part_rows_of), and where 256 rows' 32 splits would make the longest item this many positions shorter, the pass stays at 256.  us a
// layer, two rows behind 60,000 positions and 700 without, 28-layer shape: 1,133 in one pass, 748 with the first 256 rows by
// themselves; behind 30,000 884 and 693, behind 15,000 756 and 717 (40-layer shape 694 and 735).
constexpr int PREFILL_LONG_ITEM = 1300;
static bool wants_all_splits(const sparsk_ctx *c, const std::vector<PromptGroup> &groups, int n)
{
    const sparsk_dims &d = c->dm;
    if (n <= GM_MAX_N || !c->attn_tc || !c->tc_ok || d.head_dim != TA_HD || c->attn_split > 0) return false;
    int few_len = 0, many = 0;
    for (const PromptGroup &g : groups) {
        if (g.rows * (d.n_q_heads / d.n_kv_heads) < c->attn_tc_min_q) few_len = std::max(few_len, g.len);
        else many = 1;
    }
    const int splits = (int)std::min<size_t>(AT_MAX_SPLITS, std::max<size_t>(1, part_rows_of(&d) / n));
    return many && div_up(few_len, splits) - div_up(few_len, AT_MAX_SPLITS) > PREFILL_LONG_ITEM;
}

extern "C" int sparsk_prefill(sparsk_ctx *ctx, int32_t n_seqs, const int32_t *slots, const int32_t *tokens,
                              const int32_t *offsets)
{
    if (!good(ctx)) return SPARSK_ESTATE;
    const sparsk_dims &d = ctx->dm;
    if (n_seqs < 0 || n_seqs > d.max_seqs || (n_seqs && (!slots || !tokens || !offsets)))
        return fail(ctx, SPARSK_EINVAL, "prefill: bad arguments");
    std::vector<char> seen(d.max_seqs, 0);
    long rows_left = 0;
    for (int i = 0; i < n_seqs; i++) {
        const int s = slots[i];
        if (s < 0 || s >= d.max_seqs || seen[s]) return fail(ctx, SPARSK_EINVAL, "prefill: slot %d invalid or repeated", s);
        seen[s] = 1;
        const long n = (long)offsets[i + 1] - offsets[i];
        if (n < 0 || offsets[i] < 0) return fail(ctx, SPARSK_EINVAL, "prefill: offsets must not decrease");
        if (ctx->h_pend[s]) return fail(ctx, SPARSK_ESTATE, "prefill: slot %d has pending positions", s);
        if (ctx->h_len[s] + n > d.max_seq_len) return fail(ctx, SPARSK_ECAPACITY, "prefill: slot %d would hold %ld > %d positions", s, ctx->h_len[s] + n, d.max_seq_len);
        rows_left += n;
    }
    // Passes of up to `chunk` rows, filled from the prompts in order: the end of one prompt, whole
    // short ones and the beginning of the next share a pass (each a group of its own), so that only
    // the last pass of the call runs with fewer rows.
    const int chunk = std::min(d.prefill_rows, ctx->cap_rows), G_heads = d.n_q_heads / d.n_kv_heads;
    int *const r_slot = ctx->pf_rows, *const r_pos = r_slot + ctx->cap_rows, *const r_g0 = r_pos + ctx->cap_rows,
              *const r_gn = r_g0 + d.max_seqs, *const r_cnt = r_gn + d.max_seqs;
    PromptPieces in;
    std::vector<PromptGroup> groups;  // of a pass
    for (int i = 0, done = 0; i < n_seqs;) {
        auto next_groups = [&](int rows) {
            groups.clear();
            for (int j = i, had = done; rows > 0 && j < n_seqs; j++, had = 0) {
                const int take = std::min(rows, offsets[j + 1] - offsets[j] - had);
                if (take > 0) groups.push_back({take, ctx->h_len[slots[j]] + take});
                rows -= take;
            }
        };
        int n = 0, ng = 0, k = 0, max_grp = 1, max_len = 0, n_big = 0;  // rows, groups (k of them in `in`) of the pass
        long sum_len = 0;
        auto begin = [&](bool last) {  // the k pieces in hand
            const int rows = in.row0[k] - in.row0[0], first = ng - k, pieces = k;
            k = 0;
            return launch(ctx, prompt_begin_kernel, dim3(rows), dim3(128), 0, in, pieces, first, last, tokens, r_slot, r_pos, r_g0,
                          r_gn, r_cnt, ctx->embed, ctx->h_up, d.d_model, d.vocab_text + d.vocab_speech, ctx->sd.counts + CNT_STATUS);
        };
        int pass = prefill_pass_rows(ctx, rows_left, chunk);
        next_groups(pass);
        if (wants_all_splits(ctx, groups, pass)) next_groups(pass = GM_MAX_N);
        rows_left -= pass;
        while (i < n_seqs && n < pass) {
            const int s = slots[i], left = offsets[i + 1] - offsets[i] - done, take = std::min(pass - n, left);
            if (take > 0) {
                if (k == PP_MAX) CU(begin(false));
                const int pos0 = ctx->h_len[s];
                in.row0[k] = n;
                in.slot[k] = s;
                in.pos[k] = pos0;
                in.token[k] = offsets[i] + done;
                in.row0[++k] = n + take;
                ng++;
                max_grp = std::max(max_grp, take);
                max_len = std::max(max_len, pos0 + take);
                sum_len += pos0 + take;
                n_big += take * G_heads >= ctx->attn_tc_min_q;
                n += take;
                done += take;
                ctx->h_len[s] = pos0 + take;
            }
            if (take == left) {
                i++;
                done = 0;
            }
        }
        if (n == 0) break;
        CU(begin(true));
        RowSet rs{r_slot, r_pos, r_g0, r_gn, r_cnt, r_cnt + 1, n, ng, max_grp, max_len, n_big};
        rs.sum_len = sum_len;
        rs.prompt = groups.data();
        CU(run_layers(ctx, 1, d.n_layers, ctx->h_up, rs));
        CU(launch(ctx, prefill_len_kernel, dim3((ng + 127) / 128), dim3(128), 0, ctx->kv_len, (const int *)r_slot, (const int *)r_pos,
                  (const int *)r_g0, (const int *)r_gn, ng));
    }
    return SPARSK_OK;
}

// --------------------------------------------------------------------------- beginning and end of a step
// Input tokens of a step: on the device, or host values that ride along as kernel arguments.
struct StepTokens {
    const int32_t *dev, *host;
};

// Hands the step's arrays to the device and runs its first kernel: schedule, compaction (exit layer
// e), embedding, the parity hook's logits.
static int step_begin(sparsk_ctx *ctx, int n, const int32_t *slots, StepTokens tokens, const uint8_t *modality,
                      const int32_t *counters, const SchedParams &sp, int e)
{
    const sparsk_dims &d = ctx->dm;
    const int V = d.vocab_text + d.vocab_speech;
    StepIn in;
    const int *staged = nullptr;
    if (n <= SI_MAX) {
        for (int i = 0; i < n; i++) {
            in.slot[i] = slots[i];
            in.modality[i] = modality[i];
            in.counter[i] = counters[i];
            in.token[i] = tokens.host ? tokens.host[i] : 0;
        }
    } else {
        const int ring = ctx->stage_next;
        ctx->stage_next = (ring + 1) % STAGE_RING;
        CU(cudaEventSynchronize(ctx->stage_ev[ring]));
        int *st = ctx->stage_host[ring];
        for (int i = 0; i < n; i++) {
            st[i] = slots[i];
            st[n + i] = modality[i];
            st[2 * n + i] = counters[i];
        }
        CU(cudaMemcpyAsync(ctx->staged, st, sizeof(int) * 3 * n, cudaMemcpyHostToDevice, ctx->stream));
        CU(cudaEventRecord(ctx->stage_ev[ring], ctx->stream));
        staged = ctx->staged;
        if (tokens.host) {
            memcpy(ctx->io_host, tokens.host, sizeof(int) * n);
            CU(cudaMemcpyAsync(ctx->tok_dev, ctx->io_host, sizeof(int) * n, cudaMemcpyHostToDevice, ctx->stream));
            tokens.dev = ctx->tok_dev;
        }
    }
    const size_t n_logits = ctx->dbg_logits ? (size_t)n * V : 0;
    const int threads = std::max(256, div_up(n, 32) * 32);
    const int fill = (int)std::min<size_t>((n_logits + threads * 8 - 1) / (threads * 8), 2048);
    CU(launch(ctx, step_begin_kernel, dim3(1 + n + fill), dim3(threads), 0, ctx->sd, in, n, staged, tokens.dev, V, sp,
              (const int *)ctx->kv_len, (const int *)ctx->pend_cnt, e, d.max_seqs, ctx->embed, ctx->h_lo, d.d_model,
              ctx->dbg_logits, n_logits));
    return SPARSK_OK;
}
static int step_finish(sparsk_ctx *ctx, int n, int32_t *next_tokens, int32_t *exit_depths, int *status_out)
{
    const int threads = 128;
    CU(launch(ctx, finish_kernel, dim3(ctx->dbg_hidden ? n : div_up(n, threads)), dim3(threads), 0, ctx->sd, n, ctx->kv_len,
              ctx->pend_cnt, (int *)next_tokens, (int *)exit_depths, ctx->dm.n_layers, status_out, (const float *)ctx->h_lo,
              (const float *)ctx->h_up, ctx->dbg_hidden, ctx->dm.d_model));
    return SPARSK_OK;
}

// --------------------------------------------------------------------------- decode step, confidence-based exit
// The step of a context whose dims name a confidence modality (Sec. V-B, compared method 3).
// Depths are not known beforehand, so the host walks the layers in segments: a segment is a run
// of layers over one row set; it ends where a pending position joins (the layer after the one it
// has been carried to), where a scheduled sequence leaves, and after every layer from
// conf_start on while a confidence sequence is still running, because there its head is
// consulted: head, entropy kernel, copy of the entropies to the host, stream synchronisation,
// decision.  Pending positions carry the layer they have been filled to; a sequence's rows in a
// segment are the pending positions not yet carried through its first layer (always the newest
// ones: an older position has been carried at least as far as a newer one) followed by the
// current position, i.e. consecutive positions, one attention group.
static int decode_step_conf(sparsk_ctx *ctx, int32_t n, const int32_t *slots, StepTokens tokens, const uint8_t *modality,
                            const int32_t *counters, int32_t *next_tokens, int32_t *exit_depths, int *status_out)
{
    const sparsk_dims &d = ctx->dm;
    const int L = d.n_layers, e = d.exit_layer, B = d.max_seqs, cs = d.conf_start;
    const int V = d.vocab_text + d.vocab_speech, G_heads = d.n_q_heads / d.n_kv_heads;
    const SchedParams sp{L, e, d.refresh_period, d.refresh_phase, d.text_period > 0 ? d.text_period : d.refresh_period,
                         d.text_period > 0 ? d.text_phase : d.refresh_phase, d.text_exit};
    std::vector<char> seen(B, 0);
    std::vector<int> target(n), depth(n, 0);
    int max_len = 0;
    for (int i = 0; i < n; i++) {
        const int s = slots[i];
        if (s < 0 || s >= B || seen[s]) return fail(ctx, SPARSK_EINVAL, "decode_step: slot %d invalid or repeated", s);
        seen[s] = 1;
        if (modality[i] > 1) return fail(ctx, SPARSK_EINVAL, "decode_step: modality[%d]=%d", i, modality[i]);
        if (counters[i] < 0) return fail(ctx, SPARSK_EINVAL, "decode_step: counter[%d]=%d", i, counters[i]);
        if (ctx->h_len[s] + 1 > d.max_seq_len) return fail(ctx, SPARSK_ECAPACITY, "decode_step: slot %d is full (%d positions)", s, ctx->h_len[s]);
        const bool by_conf = (d.conf_modalities >> (modality[i] ? 1 : 0)) & 1;
        target[i] = by_conf ? 0 : scheduled_depth(modality[i], counters[i], sp);
        if (target[i] != L && (int)ctx->h_fill[s].size() + 1 > d.max_pending)
            return fail(ctx, SPARSK_ECAPACITY, "decode_step: slot %d may hold %d pending positions (max_pending %d)", s,
                        (int)ctx->h_fill[s].size() + 1, d.max_pending);
        if (target[i] && (!ctx->head_norm[target[i] - 1] || !ctx->head_proj[target[i] - 1]))
            return fail(ctx, SPARSK_ENOHEAD, "decode_step: layer %d has no exit head", target[i]);
        max_len = std::max(max_len, ctx->h_len[s] + 1);
    }
    // "e = L" keeps every head on the lower rows
    if (const int rc = step_begin(ctx, n, slots, tokens, modality, counters, sp, L)) return rc;
    const int R = ctx->cap_rows;
    size_t arena = 0;  // ints of the pinned arena used so far in this step
    auto region = [&](size_t ints) -> int * {
        if (arena + ints > ctx->conf_host_ints) return nullptr;
        int *p = ctx->conf_host + arena;
        arena += ints;
        return p;
    };
    // heads of `layer` for the listed sequences (indices into the step), text and speech apart
    auto heads = [&](int layer, const std::vector<int> &who) -> int {
        for (int mod = 0; mod < 2; mod++) {
            std::vector<int> rows;
            for (int i : who)
                if ((modality[i] ? 1 : 0) == mod) rows.push_back(i);
            if (rows.empty()) continue;
            int *hb = region(rows.size());
            if (!hb) return fail(ctx, SPARSK_ECAPACITY, "decode_step: staging arena exhausted");
            std::copy(rows.begin(), rows.end(), hb);
            CU(cudaMemcpyAsync(ctx->sd.list_row + (size_t)mod * B, hb, sizeof(int) * rows.size(), cudaMemcpyHostToDevice, ctx->stream));
            CU(cudaMemcpyAsync(ctx->sd.list_seq + (size_t)mod * B, hb, sizeof(int) * rows.size(), cudaMemcpyHostToDevice, ctx->stream));
            CU(launch(ctx, clear_keys_kernel, dim3(((int)rows.size() + 127) / 128), dim3(128), 0, ctx->sd.argmax,
                      (const int *)(ctx->sd.list_row + (size_t)mod * B), (int)rows.size()));
            CU(run_head(ctx, layer, ctx->h_lo, mod, (int)rows.size()));
        }
        return SPARSK_OK;
    };
    auto leave = [&](int i, int at) -> int {   // sequence i leaves at layer `at`
        const int s = slots[i];
        depth[i] = at;
        std::vector<int> &fill = ctx->h_fill[s];
        if (at == L) {
            fill.clear();
        } else {
            CU(cudaMemcpyAsync(ctx->pend_h + ((size_t)s * d.max_pending + fill.size()) * d.d_model, ctx->h_lo + (size_t)i * d.d_model,
                               sizeof(float) * d.d_model, cudaMemcpyDeviceToDevice, ctx->stream));
            fill.push_back(at);
        }
        return SPARSK_OK;
    };

    std::vector<int> active(n);
    for (int i = 0; i < n; i++) active[i] = i;
    ctx->conf_trace.assign((size_t)n * L, -1.f);
    int l = 1;
    while (!active.empty()) {
        // ---- where this segment ends
        int seg_end = L;
        for (int i : active) {
            seg_end = std::min(seg_end, target[i] ? target[i] : std::max(l, cs));
            for (int f : ctx->h_fill[slots[i]])
                if (f >= l) seg_end = std::min(seg_end, f);
        }
        // ---- its rows
        struct Row { int slot, pos, src, seq; };
        std::vector<Row> rows;
        std::vector<int> g_row0, g_nrows;
        int max_grp = 1, n_big = 0, seg_len = 0;
        for (int i : active) {
            const int s = slots[i];
            const std::vector<int> &fill = ctx->h_fill[s];
            const int P = (int)fill.size();
            int j0 = 0;
            while (j0 < P && fill[j0] >= l) j0++;   // carried through layer l already
            g_row0.push_back((int)rows.size());
            g_nrows.push_back(P - j0 + 1);
            for (int j = j0; j < P; j++) rows.push_back({s, ctx->h_len[s] - P + j, j, i});
            rows.push_back({s, ctx->h_len[s], -1, i});
            max_grp = std::max(max_grp, P - j0 + 1);
            n_big += (P - j0 + 1) * G_heads >= ctx->attn_tc_min_q;
            seg_len = std::max(seg_len, ctx->h_len[s] + 1);
        }
        const int m = (int)rows.size(), ng = (int)active.size();
        if (m > R) return fail(ctx, SPARSK_ECAPACITY, "decode_step: %d rows exceed capacity %d", m, R);
        if (m == n && ng == n) {
            // nothing but the step's own positions, in order: the lower rows as they stand
            RowSet lo{ctx->sd.slot, ctx->sd.lo_pos, ctx->sd.lo_grp_row0, ctx->sd.lo_grp_nrows, ctx->sd.counts + CNT_NSEQ,
                      ctx->sd.counts + CNT_NSEQ, n, n, 1, seg_len};
            CU(run_layers(ctx, l, seg_end, ctx->h_lo, lo));
        } else {
            int *hb = region(4 * (size_t)R + 2 * (size_t)B + 2);
            if (!hb) return fail(ctx, SPARSK_ECAPACITY, "decode_step: staging arena exhausted");
            int *h_slot = hb, *h_pos = hb + R, *h_src = hb + 2 * R, *h_seq = hb + 3 * R, *h_g0 = hb + 4 * R, *h_gn = h_g0 + B,
                *h_cnt = h_gn + B;
            for (int k = 0; k < m; k++) {
                h_slot[k] = rows[k].slot; h_pos[k] = rows[k].pos; h_src[k] = rows[k].src; h_seq[k] = rows[k].seq;
            }
            for (int k = 0; k < ng; k++) {
                h_g0[k] = g_row0[k];
                h_gn[k] = g_nrows[k];
            }
            h_cnt[0] = ng;
            h_cnt[1] = m;
            int *dv = ctx->conf_rows_dev;
            CU(cudaMemcpyAsync(dv, hb, sizeof(int) * (4 * (size_t)R + 2 * (size_t)B + 2), cudaMemcpyHostToDevice, ctx->stream));
            int *d_slot = dv, *d_pos = dv + R, *d_src = dv + 2 * R, *d_seq = dv + 3 * R, *d_g0 = dv + 4 * R, *d_gn = d_g0 + B,
                *d_cnt = d_gn + B;
            CU(launch(ctx, rows_move_kernel, dim3(m), dim3(128), 0, ctx->h_up, ctx->h_lo, ctx->pend_h, (const int *)d_slot,
                      (const int *)d_seq, (const int *)d_src, m, d.d_model, d.max_pending, 1));
            RowSet up{d_slot, d_pos, d_g0, d_gn, d_cnt, d_cnt + 1, m, ng, max_grp, seg_len, n_big};
            CU(run_layers(ctx, l, seg_end, ctx->h_up, up));
            CU(launch(ctx, rows_move_kernel, dim3(m), dim3(128), 0, ctx->h_up, ctx->h_lo, ctx->pend_h, (const int *)d_slot,
                      (const int *)d_seq, (const int *)d_src, m, d.d_model, d.max_pending, 0));
        }
        for (int i : active)   // the pending positions that took part have been carried to seg_end
            for (int &f : ctx->h_fill[slots[i]])
                if (f < seg_end) f = seg_end;
        // ---- who leaves after layer seg_end
        std::vector<int> leaving, asking;
        for (int i : active) {
            if (seg_end == L || target[i] == seg_end) leaving.push_back(i);
            else if (!target[i] && seg_end >= cs) asking.push_back(i);
        }
        if (!leaving.empty()) {
            const int rc = heads(seg_end, leaving);
            if (rc != SPARSK_OK) return rc;
        }
        if (!asking.empty()) {
            int rc = heads(seg_end, asking);
            if (rc != SPARSK_OK) return rc;
            int *hb = region(2 * asking.size());
            if (!hb) return fail(ctx, SPARSK_ECAPACITY, "decode_step: staging arena exhausted");
            for (size_t k = 0; k < asking.size(); k++) {
                hb[k] = asking[k];
                hb[asking.size() + k] = modality[asking[k]] ? 1 : 0;
            }
            CU(cudaMemcpyAsync(ctx->conf_list_dev, hb, sizeof(int) * 2 * asking.size(), cudaMemcpyHostToDevice, ctx->stream));
            CU(launch(ctx, entropy_kernel, dim3((unsigned)asking.size()), dim3(1024), 0, (const float *)head_logits(ctx),
                      (const int *)ctx->conf_list_dev, (const int *)(ctx->conf_list_dev + asking.size()), (int)asking.size(), V,
                      d.vocab_text, ctx->conf_ent_dev));
            CU(cudaMemcpyAsync(ctx->conf_ent_host, ctx->conf_ent_dev, sizeof(float) * asking.size(), cudaMemcpyDeviceToHost, ctx->stream));
            CU(cudaStreamSynchronize(ctx->stream));
            for (size_t k = 0; k < asking.size(); k++) {
                ctx->conf_trace[(size_t)asking[k] * L + seg_end] = ctx->conf_ent_host[k];
                if (ctx->conf_ent_host[k] < d.conf_threshold) leaving.push_back(asking[k]);
            }
        }
        for (int i : leaving) {
            const int rc = leave(i, seg_end);
            if (rc != SPARSK_OK) return rc;
            active.erase(std::find(active.begin(), active.end(), i));
        }
        l = seg_end + 1;
    }
    // ---- outputs and state
    int *hb = region(n);
    if (!hb) return fail(ctx, SPARSK_ECAPACITY, "decode_step: staging arena exhausted");
    std::copy(depth.begin(), depth.end(), hb);
    CU(cudaMemcpyAsync(ctx->sd.depth, hb, sizeof(int) * n, cudaMemcpyHostToDevice, ctx->stream));
    if (const int rc = step_finish(ctx, n, next_tokens, exit_depths, status_out)) return rc;
    for (int i = 0; i < n; i++) {
        ctx->h_len[slots[i]] += 1;
        ctx->h_pend[slots[i]] = (int)ctx->h_fill[slots[i]].size();
    }
    CU(cudaStreamSynchronize(ctx->stream));  // the pinned arena is free again
    return SPARSK_OK;
}

// --------------------------------------------------------------------------- decode step
static int decode_step(sparsk_ctx *ctx, int32_t n, const int32_t *slots, StepTokens tokens, const uint8_t *modality,
                       const int32_t *counters, int32_t *next_tokens, int32_t *exit_depths, int *status_out)
{
    const sparsk_dims &d = ctx->dm;
    const int L = d.n_layers, e = d.exit_layer, B = d.max_seqs;
    const SchedParams sp{L, e, d.refresh_period, d.refresh_phase, d.text_period > 0 ? d.text_period : d.refresh_period,
                         d.text_period > 0 ? d.text_phase : d.refresh_phase, d.text_exit};
    if (n < 1 || n > B || !slots || !(tokens.dev || tokens.host) || !modality || !counters || !next_tokens || !exit_depths)
        return fail(ctx, SPARSK_EINVAL, "decode_step: bad arguments (n=%d)", n);
    if (d.conf_modalities) return decode_step_conf(ctx, n, slots, tokens, modality, counters, next_tokens, exit_depths, status_out);
    // ---- host mirror of the schedule: validates, and sizes the launches
    std::vector<char> seen(B, 0);
    int n_list[4] = {0, 0, 0, 0};
    int m_up = 0, n_grp = 0, max_grp = 1, max_len_lo = 0, max_len_up = 0, n_big = 0;
    long sum_len_lo = 0, sum_len_up = 0;
    const int G_heads = d.n_q_heads / d.n_kv_heads;
    for (int i = 0; i < n; i++) {
        const int s = slots[i];
        if (s < 0 || s >= B || seen[s]) return fail(ctx, SPARSK_EINVAL, "decode_step: slot %d invalid or repeated", s);
        seen[s] = 1;
        if (modality[i] > 1) return fail(ctx, SPARSK_EINVAL, "decode_step: modality[%d]=%d", i, modality[i]);
        if (counters[i] < 0) return fail(ctx, SPARSK_EINVAL, "decode_step: counter[%d]=%d", i, counters[i]);
        if (ctx->h_len[s] + 1 > d.max_seq_len) return fail(ctx, SPARSK_ECAPACITY, "decode_step: slot %d is full (%d positions)", s, ctx->h_len[s]);
        const int depth = scheduled_depth(modality[i], counters[i], sp);
        const bool full = depth == L;
        if (!full && ctx->h_pend[s] + 1 > d.max_pending)
            return fail(ctx, SPARSK_ECAPACITY, "decode_step: slot %d would hold %d pending positions (max_pending %d)", s, ctx->h_pend[s] + 1, d.max_pending);
        n_list[(full ? 2 : 0) + (modality[i] ? 1 : 0)]++;
        max_len_lo = std::max(max_len_lo, ctx->h_len[s] + 1);
        sum_len_lo += ctx->h_len[s] + 1;
        if (full && e < L) {
            sum_len_up += ctx->h_len[s] + 1;
            m_up += ctx->h_pend[s] + 1;
            n_grp++;
            max_grp = std::max(max_grp, ctx->h_pend[s] + 1);
            n_big += (ctx->h_pend[s] + 1) * G_heads >= ctx->attn_tc_min_q;
            max_len_up = std::max(max_len_up, ctx->h_len[s] + 1);
        }
    }
    if ((n_list[0] + n_list[1]) && (!ctx->head_norm[e - 1] || !ctx->head_proj[e - 1]))
        return fail(ctx, SPARSK_ENOHEAD, "decode_step: layer %d has no exit head", e);
    if (m_up > ctx->cap_rows) return fail(ctx, SPARSK_ECAPACITY, "decode_step: %d upper rows exceed capacity %d", m_up, ctx->cap_rows);

    // ---- schedule, compaction, embedding
    const int V = d.vocab_text + d.vocab_speech;
    if (const int rc = step_begin(ctx, n, slots, tokens, modality, counters, sp, e)) return rc;
    // ---- lower pass: layers 1..e over all sequences
    RowSet lo{ctx->sd.slot, ctx->sd.lo_pos, ctx->sd.lo_grp_row0, ctx->sd.lo_grp_nrows, ctx->sd.counts + CNT_NSEQ,
              ctx->sd.counts + CNT_NSEQ, n, n, 1, max_len_lo};
    lo.sum_len = sum_len_lo;
    CU(run_layers(ctx, 1, e, ctx->h_lo, lo));
    // ---- early exits keep h^(e); the upper pass gathers its rows
    const int n_early = n_list[0] + n_list[1];
    if (n_early || m_up)
        CU(launch(ctx, exit_rows_kernel, dim3((n_early ? n : 0) + m_up), dim3(128), 0, ctx->sd, (const float *)ctx->h_lo,
                  ctx->pend_h, (const int *)ctx->pend_cnt, ctx->h_up, n_early ? n : 0, d.d_model, L, d.max_pending));
    // ---- early exits read the token from g_e
    for (int l = 0; l < 2; l++)
        if (n_list[l]) CU(run_head(ctx, e, ctx->h_lo, l, n_list[l]));
    // ---- upper pass: pending and current positions of full-depth sequences through e+1..L
    const float *h_full = ctx->h_lo;
    if (m_up) {
        RowSet up{ctx->sd.up_slot, ctx->sd.up_pos, ctx->sd.up_grp_row0, ctx->sd.up_grp_nrows, ctx->sd.counts + CNT_NGRP,
                  ctx->sd.counts + CNT_MUP, m_up, n_grp, max_grp, max_len_up, n_big};
        up.sum_len = sum_len_up;
        // Layer L gives the pending rows nothing but their K/V: nothing reads their h^(L).  When the
        // step has pending rows and the rest of the layer is cheaper on one row per sequence
        // (attention over long prefixes, projections with enough rows to be tensor-bound), the
        // layer's back half runs on the current rows alone.
        const int qd = d.n_q_heads * d.head_dim;
        const bool persistent = use_mega(ctx, m_up);
        const bool trim = m_up > n_grp && !persistent &&
                          (ctx->trim_last == 2 || (ctx->trim_last == 1 && use_tc(ctx, n_grp)));
        if (!trim) {
            CU(run_layers(ctx, e + 1, L, ctx->h_up, up));
        } else {
            CU(run_layers(ctx, e + 1, L - 1, ctx->h_up, up));
            ctx->route_layers[use_tc(ctx, m_up) ? 1 : 2] += 1;
            CU(run_layer_front(ctx, L, ctx->h_up, up));
            CU(launch(ctx, take_current_kernel, dim3(n_grp), dim3(256), 0, ctx->sd, (const float *)ctx->h_up,
                      (const float *)ctx->qbuf, ctx->h_last, ctx->q_last, ctx->last_slot, ctx->last_pos, d.d_model, qd));
            RowSet last{ctx->last_slot, ctx->last_pos, ctx->sd.lo_grp_row0, ctx->sd.lo_grp_nrows, ctx->sd.counts + CNT_NGRP,
                        ctx->sd.counts + CNT_NGRP, n_grp, n_grp, 1, max_len_up, 0, ctx->q_last};
            last.sum_len = sum_len_up;
            last.rows_late = true;
            CU(run_layer_back(ctx, L, ctx->h_last, last));
            CU(launch(ctx, put_current_kernel, dim3(n_grp), dim3(256), 0, ctx->sd, (const float *)ctx->h_last, ctx->h_up,
                      d.d_model));
        }
        h_full = ctx->h_up;
    }
    for (int l = 2; l < 4; l++)
        if (n_list[l]) CU(run_head(ctx, L, h_full, l, n_list[l]));
    if (ctx->samp_uniforms) {
        // replace the arg max by a draw from the nucleus of the same logits (Sec. V-A)
        SampleArgs sa{};
        sa.logits = head_logits(ctx); sa.uniforms = ctx->samp_uniforms;
        sa.modality = ctx->sd.modality; sa.key_out = ctx->sd.argmax; sa.token_out = nullptr;
        sa.V = V; sa.Vt = d.vocab_text; sa.Vs = d.vocab_speech;
        sa.inv_temperature = 1.f / ctx->samp_temperature; sa.top_p = ctx->samp_top_p;
        const bool timed = (ctx->time_class == KC_HEAD || ctx->time_class == KC_ALL) && ctx->tev_used + 2 <= ctx->tev.size();
        if (timed) {
            ctx->tev_class[ctx->tev_used / 2] = KC_HEAD;
            cudaEventRecord(ctx->tev[ctx->tev_used++], ctx->stream);
        }
        CU(launch_nucleus_sample(sa, n, n_list[0] + n_list[2] > 0, n_list[1] + n_list[3] > 0, ctx->stream, ctx->pdl != 0,
                                 &ctx->launches));
        if (timed) cudaEventRecord(ctx->tev[ctx->tev_used++], ctx->stream);
    }
    if (const int rc = step_finish(ctx, n, next_tokens, exit_depths, status_out)) return rc;
    // ---- host mirror follows
    for (int i = 0; i < n; i++) {
        const int s = slots[i];
        const int depth = scheduled_depth(modality[i], counters[i], sp);
        ctx->h_len[s] += 1;
        ctx->h_pend[s] = (depth == L) ? 0 : ctx->h_pend[s] + 1;
    }
    return SPARSK_OK;
}

extern "C" int sparsk_decode_step(sparsk_ctx *ctx, int32_t n, const int32_t *slots, const int32_t *token_ids,
                                  const uint8_t *modality, const int32_t *counters, int32_t *next_tokens,
                                  int32_t *exit_depths)
{
    if (!good(ctx)) return SPARSK_ESTATE;
    return decode_step(ctx, n, slots, {token_ids, nullptr}, modality, counters, next_tokens, exit_depths, nullptr);
}

extern "C" int sparsk_decode_step_host(sparsk_ctx *ctx, int32_t n, const int32_t *slots, const int32_t *token_ids,
                                       const uint8_t *modality, const int32_t *counters, int32_t *next_tokens,
                                       int32_t *exit_depths)
{
    if (!good(ctx)) return SPARSK_ESTATE;
    if (n < 1 || n > ctx->dm.max_seqs || !token_ids || !next_tokens || !exit_depths)
        return fail(ctx, SPARSK_EINVAL, "decode_step_host: bad arguments (n=%d)", n);
    // the tokens are host data here, so their range is checked like every other host argument:
    // before anything is enqueued, leaving all state as it was
    const int V = ctx->dm.vocab_text + ctx->dm.vocab_speech;
    for (int i = 0; i < n; i++)
        if (token_ids[i] < 0 || token_ids[i] >= V)
            return fail(ctx, SPARSK_EINVAL, "decode_step_host: token_ids[%d]=%d is outside the vocabulary [0, %d)", i, token_ids[i], V);
    // The tokens ride along as kernel arguments (or through the pinned buffer, beyond SI_MAX
    // sequences), and the step's last kernel writes the results and the status word straight into
    // pinned memory: no copies before or behind the step, one wait.
    const int B = ctx->dm.max_seqs;
    int *io = ctx->io_host;
    const int rc = decode_step(ctx, n, slots, {nullptr, token_ids}, modality, counters, io + B, io + 2 * B, io + 3 * B);
    if (rc != SPARSK_OK) return rc;
    CU(cudaStreamSynchronize(ctx->stream));
    memcpy(next_tokens, io + B, sizeof(int) * n);
    memcpy(exit_depths, io + 2 * B, sizeof(int) * n);
    return act_on_status(ctx, io[3 * B]);
}
