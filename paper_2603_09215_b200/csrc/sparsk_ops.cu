// Stand-alone entry points for single kernels of the decode path (C ABI in include/sparsk.h).
// They run exactly the kernels a decode step runs, on caller-described inputs, so that one
// stage can be driven, checked and profiled on its own.
#include <algorithm>
#include <cstdint>

#include "../../include/sparsk.h"
#include "sparsk_attn.cuh"
#include "sparsk_sample.cuh"
#include "sparsk_step.cuh"

using namespace sparsk;

namespace {
size_t up256(size_t v) { return (v + 255) / 256 * 256; }
}  // namespace

static bool attn_args_ok(const sparsk_attn_args *a)
{
    if (!a || !a->q || !a->k_cache || !a->v_cache || !a->out || !a->row_slot || !a->row_pos || !a->grp_row0 ||
        !a->grp_nrows)
        return false;
    if (a->n_rows < 1 || a->n_groups < 1 || a->n_groups > a->n_rows || a->max_grp_rows < 1 ||
        a->max_grp_rows > a->n_rows)
        return false;
    if (a->n_q_heads < 1 || a->n_kv_heads < 1 || a->n_q_heads % a->n_kv_heads) return false;
    if (a->head_dim != 64 && a->head_dim != 128) return false;
    if (a->cache_len < 1 || a->n_slots < 1 || a->max_len < 1 || a->max_len > a->cache_len) return false;
    return true;
}

extern "C" size_t sparsk_attention_scratch_bytes(int32_t n_rows, int32_t n_q_heads, int32_t head_dim)
{
    if (n_rows < 1 || n_q_heads < 1 || (head_dim != 64 && head_dim != 128)) return 0;
    const size_t cells = (size_t)n_rows * n_q_heads * AT_MAX_SPLITS;
    return 256 + up256(cells * head_dim * sizeof(float)) + up256(cells * sizeof(float2));
}

// The two launches follow each other as in a decode step: the merge may be resident before the
// partials are complete and waits for them itself.
template <class... KArgs, class... Args>
static cudaError_t launch_dependent(cudaStream_t st, void (*kern)(KArgs...), dim3 grid, int block, size_t smem, Args... args)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, KArgs(args)...);
}

static int n_sm_here()
{
    static PerDevice<int> sms;
    int &n = sms.here();
    if (n == 0) {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) n = 0;
    }
    return n;
}

// Shared by the entry points of this library that run the two attention kernels outside a
// context: `scratch` holds an item counter, then the split partials.
int sparsk_attention_launch(const sparsk_attn_args *p, char *scratch, cudaStream_t st)
{
    const int n_sm = n_sm_here();
    if (n_sm == 0) return SPARSK_ECUDA;
    const size_t cells = (size_t)p->n_rows * p->n_q_heads * AT_MAX_SPLITS;
    AttnArgs a{};
    a.q = (const bf16 *)p->q; a.kc = (const kv_t *)p->k_cache; a.vc = (const kv_t *)p->v_cache;
    a.grp_row0 = p->grp_row0; a.grp_nrows = p->grp_nrows; a.row_slot = p->row_slot; a.row_pos = p->row_pos;
    a.part_o = reinterpret_cast<float *>(scratch + 256);
    a.part_ml = reinterpret_cast<float2 *>(scratch + 256 + up256(cells * p->head_dim * sizeof(float)));
    a.out = (bf16 *)p->out;
    a.Hq = p->n_q_heads; a.Hkv = p->n_kv_heads; a.S = p->cache_len; a.n_slots = p->n_slots; a.n_rows = p->n_rows;
    a.nq_min = 0; a.nq_max = 1 << 30;
    const int warp_ctas = n_sm * attn_warp_ctas_per_sm(p->head_dim, AW_NST);
    // Only a bound on the prefixes is known here: with several groups they are taken to be half as long
    // on average.  That suits ragged lengths and costs uniform ones.  us a call back to back, planned
    // for the bound / for half of it (28 query heads of 128, 4 kv heads, unless given): 48 groups of 200 to
    // 3,000 positions, every third of four rows 63.1 / 59.8, all of one row 46.4 / 45.2, one of 3,000
    // among 47 of 100 25.6 / 23.1, 64 of 500 to 4,000 and four rows (32 heads, 2 kv heads) 126.0 / 116.6;
    // against that 48 of 3,000 each 63.5 / 67.0, with four rows 100.7 / 119.0, 32 of 2,048 and eight rows (32
    // heads, 8 kv heads) 96.0 / 115.9.  (A fifth: 63 for the first.)
    const AttnPlan pl = attn_plan(warp_ctas * AW_WARPS, p->n_groups, p->max_grp_rows, p->n_q_heads / p->n_kv_heads,
                                  p->n_kv_heads, p->max_len, 0, p->n_groups > 1 ? (long)p->n_groups * p->max_len / 2 : 0);
    a.n_qblk = pl.n_qblk; a.split_len = pl.split_len; a.n_splits = pl.n_splits;
    a.max_groups = p->n_groups;
    const long n_items = (long)p->n_groups * pl.n_qblk * p->n_kv_heads * pl.n_splits;
    const int grid = (int)std::max<long>(1, std::min<long>(warp_ctas, (n_items + AW_WARPS - 1) / AW_WARPS));
    AttnWarpFn fn;
    if (attn_warp_fn(p->head_dim, AW_NST, &fn) != cudaSuccess) return SPARSK_ECUDA;
    if (n_items > (long)grid * AW_WARPS && n_items < (1L << 31)) {  // items beyond the warps' first ones are drawn
        if (cudaMemsetAsync(scratch, 0, sizeof(unsigned), st) != cudaSuccess) return SPARSK_ECUDA;
        a.ticket = reinterpret_cast<unsigned *>(scratch);
    }
    cudaError_t e = launch_dependent(st, fn, dim3(grid), AW_WARPS * 32, AW_WARPS * attn_warp_bytes(p->head_dim, AW_NST), a);
    dim3 merge_grid;
    const AttnMergeFn merge = attn_merge_fn(p->head_dim, a.n_splits, p->n_rows, p->n_q_heads, &merge_grid);
    if (e == cudaSuccess) e = launch_dependent(st, merge, merge_grid, MG_THREADS, 0, a, (const int *)nullptr);
    return e == cudaSuccess ? SPARSK_OK : SPARSK_ECUDA;
}

extern "C" int sparsk_attention(const sparsk_attn_args *args, void *scratch, size_t scratch_bytes, void *cuda_stream)
{
    if (!attn_args_ok(args) || !scratch || ((uintptr_t)scratch % 256)) return SPARSK_EINVAL;
    if (scratch_bytes < sparsk_attention_scratch_bytes(args->n_rows, args->n_q_heads, args->head_dim))
        return SPARSK_EINVAL;
    return sparsk_attention_launch(args, (char *)scratch, (cudaStream_t)cuda_stream);
}

extern "C" int sparsk_nucleus_sample(const float *logits, const float *uniforms, const int32_t *modality, int32_t n,
                                     int32_t vocab_text, int32_t vocab_speech, float temperature, float top_p,
                                     int32_t *tokens, void *cuda_stream)
{
    if (!logits || !uniforms || !modality || !tokens) return SPARSK_EINVAL;
    if (n < 1 || vocab_text < 1 || vocab_speech < 0 || vocab_text > SP_MAX_RANGE || vocab_speech > SP_MAX_RANGE)
        return SPARSK_EINVAL;
    if (!(temperature > 0.f) || !(temperature < INFINITY) || !(top_p > 0.f) || !(top_p <= 1.f)) return SPARSK_EINVAL;
    SampleArgs a{};
    a.logits = logits; a.uniforms = uniforms; a.modality = modality;
    a.key_out = nullptr; a.token_out = tokens;
    a.V = vocab_text + vocab_speech; a.Vt = vocab_text; a.Vs = vocab_speech;
    a.inv_temperature = 1.f / temperature; a.top_p = top_p;
    return launch_nucleus_sample(a, n, true, vocab_speech > 0, (cudaStream_t)cuda_stream, false, nullptr) == cudaSuccess
               ? SPARSK_OK
               : SPARSK_ECUDA;
}
