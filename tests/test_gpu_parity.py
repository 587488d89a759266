"""GPU parity: the CUDA library through its C ABI against the C oracle, element by element."""
import numpy as np
import pytest
import torch

from paper_2603_09215_b200 import synth

pytestmark = pytest.mark.gpu

MICRO64 = dict(n_layers=3, d_model=136, n_q_heads=6, n_kv_heads=2, head_dim=64, d_ffn=200,
               vocab_text=301, vocab_speech=99, rms_eps=1e-6, rope_base=10000.0)
MICRO256 = dict(n_layers=3, d_model=256, n_q_heads=4, n_kv_heads=2, head_dim=64, d_ffn=512,
                vocab_text=301, vocab_speech=99, rms_eps=1e-6, rope_base=10000.0)


@pytest.fixture(scope="module")
def util():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from tests import parity_util
    return parity_util


def test_config1_tiny_full_run(util):
    """Workload 1 in full: 32-token prompt, 96 steps, 2 text : 4 speech, e=2, K=3."""
    wl = synth.WORKLOADS["cfg1_tiny_b1"]
    dims = synth.model_dims("tiny", wl["exit_layer"], wl["refresh_period"], wl["refresh_phase"])
    w = synth.make_weights(dims, seed=0)
    prompt = synth.make_prompts(dims, 1, 32, 32)[0]
    P = util.Pair(dims, w, 1, 32 + 96 + 1, wl["refresh_period"] - 1)
    P.prefill([prompt])
    P.check_cache(0, range(1, 5), 31)
    depths = []
    for g in range(wl["steps"]):
        m, c = synth.interleave(g, wl["n_text"], wl["n_speech"])
        ref, _, dep = P.step([m], [c])
        depths.append(int(dep[0]))
        if ref[0]["depth"] == 4:       # after a full-depth step the whole cache is complete
            P.check_cache(0, range(1, 5), 32 + g)
    sp = [d for g, d in enumerate(depths) if synth.interleave(g, 2, 4)[0] == 1]
    assert sp[:4] == [4, 2, 2, 4] and sum(sp) / len(sp) == 3.0
    assert P.stats["tok_checked"] > 40, P.stats
    print("cfg1", P.stats)
    P.close()


@pytest.mark.parametrize("min_rows", [3, 1])
@pytest.mark.parametrize("e,K,r,nt,ns", [(1, 2, 0, 1, 4), (2, 4, 1, 2, 7), (3, 2, 0, 1, 4), (2, 1, 0, 1, 4),
                                          (1, 5, 4, 0, 9)])
def test_odd_shapes_and_schedules(util, e, K, r, nt, ns, min_rows):
    """head_dim 64, 3 query heads per kv head, dimensions that are not multiples of the 256-wide
    chunks, vocabulary ranges that are not multiples of the row groups; several (e, K, r)."""
    dims = synth.model_dims(MICRO64, e, K, r)
    w = synth.make_weights(dims, seed=5)
    prompt = synth.make_prompts(dims, 1, 37, 37, seed=7)[0]
    P = util.Pair(dims, w, 1, 128, 2 * K, prefill_rows=16, options={"gemm_min_rows": min_rows})
    P.prefill([prompt])
    for g in range(40):
        m, c = synth.interleave(g, nt, ns)
        P.step([m], [c])
    P.check_cache(0, range(1, 4), P.g.slot_state(0)[0] - P.g.slot_state(0)[1])
    P.close()


@pytest.mark.parametrize("min_rows,trim", [(3, 1), (1, 2), (1 << 30, 2), (3, 0), (3, 2)])
def test_heterogeneous_batch_matches_per_sequence_oracle(util, min_rows, trim):
    """Batch of 7 with random interleave phases and counter offsets and ragged prompts, so every
    step mixes text, early-exit and refresh rows; sequences stay independent.  Run with the
    default hand-over between the small-batch and the tensor-core path (3 rows), with every
    projection on the tensor cores, and with every projection on the small-batch path; and with the pending rows leaving
    the last layer after its K/V projection (trim 2: always, 1: when it pays, 0: never), which
    must change nothing: the cache of every layer is compared below."""
    dims = synth.model_dims("tiny", 2, 4, 0)
    w = synth.make_weights(dims, seed=0)
    B = 7
    prompts = synth.make_prompts(dims, B, 9, 70, seed=4)
    phi, off = synth.make_phases(B, 1, 4, 4, True, seed=8)
    P = util.Pair(dims, w, B, 70 + 64, 3, prefill_rows=24, options={"gemm_min_rows": min_rows, "trim_last_layer": trim})
    P.prefill(prompts)
    mixed = 0
    for g in range(48):
        mc = [synth.interleave(g, 1, 4, int(p), int(o)) for p, o in zip(phi, off)]
        ref, _, dep = P.step([m for m, _ in mc], [c for _, c in mc])
        mixed += len(set(int(x) for x in dep)) > 1
    assert mixed > 20
    for s in range(B):
        ln, pend = P.g.slot_state(s)
        P.check_cache(s, range(1, 3), ln)          # lower layers are always complete
        P.check_cache(s, range(3, 5), ln - pend)   # upper layers up to the last full step
    print("hetero", P.stats)
    P.close()


MICRO128 = dict(n_layers=3, d_model=192, n_q_heads=8, n_kv_heads=1, head_dim=128, d_ffn=320,
                vocab_text=211, vocab_speech=77, rms_eps=1e-6, rope_base=10000.0)


@pytest.mark.parametrize("min_q,split", [(33, 0), (1, 0), (1, 64)])
def test_tensor_core_attention_for_blocks_of_query_vectors(util, min_q, split):
    """head_dim 128 with eight query heads per kv head: flushes of five pending rows + current
    (48 query vectors), prefill chunks of 24 rows (192 query vectors = two blocks of 128) and,
    with min_q = 1, single rows too go through the tcgen05 attention kernel; with 64-position
    splits a pass has several KV splits and ragged last tiles."""
    dims = synth.model_dims(MICRO128, 1, 6, 0)
    w = synth.make_weights(dims, seed=3)
    B = 3
    prompts = synth.make_prompts(dims, B, 70, 150, seed=12)
    P = util.Pair(dims, w, B, 150 + 64, 5, prefill_rows=24,
                  options={"attn_tc_min_q": min_q, "attn_split": split})
    P.prefill(prompts)
    for s in range(B):
        P.check_cache(s, range(1, 4), len(prompts[s]) - 1)
    phases = [0, 3, 5]
    for g in range(30):
        mc = [synth.interleave(g, 1, 6, ph) for ph in phases]
        P.step([m for m, _ in mc], [c for _, c in mc])
    for s in range(B):
        ln, pend = P.g.slot_state(s)
        P.check_cache(s, range(1, 2), ln)
        P.check_cache(s, range(2, 4), ln - pend)
    print("tc attention", P.stats)
    P.close()


def test_subset_of_slots_and_slot_reuse(util):
    """Steps may name any subset of slots in any order; a reset slot starts over."""
    dims = synth.model_dims("tiny", 2, 3, 0)
    w = synth.make_weights(dims, seed=0)
    prompts = synth.make_prompts(dims, 3, 12, 20, seed=2)
    P = util.Pair(dims, w, 3, 96, 2)
    P.prefill(prompts)
    for g in range(6):
        P.step([1, 1, 1], [g % 4] * 3)
    for g in range(6):
        P.step([1, 0], [g % 4, 0], slots=[2, 0])
    P.step([0], [0], slots=[1])
    # reuse slot 1 for a new sequence
    P.g.reset_slot(1)
    P.os[1] = P.om.new_seq(2)
    newp = synth.make_prompts(dims, 1, 15, 15, seed=9)[0]
    P.g.prefill([1], [newp[:-1]])
    P.os[1].prefill(newp[:-1])
    P.next_in[1] = int(newp[-1])
    for g in range(8):
        P.step([1, 1, 1], [g % 4] * 3, slots=[1, 2, 0])
    P.close()


def test_imported_cache_long_context(util):
    """A long synthetic cache (several KV splits and tiles, ragged tail) loaded into both sides."""
    dims = synth.model_dims("tiny", 2, 4, 0)
    w = synth.make_weights(dims, seed=0)
    n = 1000 + 37
    k, v = synth.synth_kv(dims, n, seed=6)
    P = util.Pair(dims, w, 2, n + 40, 3)
    from oracle.bruteforce import bf16_to_f64
    for layer in range(1, 5):
        kt = torch.from_numpy(k[layer - 1].view(np.int16)).cuda().view(torch.bfloat16).to(torch.float16)
        vt = torch.from_numpy(v[layer - 1].view(np.int16)).cuda().view(torch.bfloat16).to(torch.float16)
        for s in range(2):
            P.g.import_kv(s, layer, 0, kt, vt)
        kf, vf = bf16_to_f64(k[layer - 1]), bf16_to_f64(v[layer - 1])
        for s in range(2):
            for p in range(n):
                P.os[s].set_kv(layer, p, kf[p], vf[p])
    for s in range(2):
        P.g.set_len(s, n)
        P.os[s].set_len(n)
    P.next_in = [3, 1030]
    for g in range(12):
        mc = [synth.interleave(g, 1, 4, ph, 0) for ph in (0, 2)]
        P.step([m for m, _ in mc], [c for _, c in mc])
    print("long", P.stats)
    P.close()


def test_host_step_and_error_codes(util):
    from paper_2603_09215_b200 import binding
    dims = synth.model_dims("tiny", 2, 3, 0)
    w = synth.make_weights(dims, seed=0, head_layers=[2, 4])
    P = util.Pair(dims, w, 2, 40, 1)
    prompts = synth.make_prompts(dims, 2, 10, 10, seed=3)
    P.prefill(prompts)
    nt, dp = np.zeros(2, np.int32), np.zeros(2, np.int32)
    ref = [P.os[s].decode_step(P.next_in[s], 1, 0) for s in range(2)]
    P.g.decode_step_host([0, 1], P.next_in, [1, 1], [0, 0], nt, dp)
    assert list(dp) == [4, 4]
    for s in range(2):
        if ref[s]["margin"] > util.MARGIN:
            assert nt[s] == ref[s]["token"]
    before = [P.g.slot_state(s) for s in range(2)]
    with pytest.raises(binding.SparskError) as ei:      # repeated slot
        P.g.decode_step_host([0, 0], [1, 1], [1, 1], [1, 1], nt, dp)
    assert ei.value.code == binding.EINVAL
    P.g.decode_step_host([0, 1], [5, 6], [1, 1], [1, 1], nt, dp)           # early exit: 1 pending
    assert list(dp) == [2, 2]
    with pytest.raises(binding.SparskError) as ei:      # a second pending position does not fit
        P.g.decode_step_host([0, 1], [5, 6], [1, 1], [2, 2], nt, dp)
    assert ei.value.code == binding.ECAPACITY
    assert [P.g.slot_state(s) for s in range(2)] == [(b[0] + 1, 1) for b in before]
    before = [P.g.slot_state(s) for s in range(2)]
    with pytest.raises(binding.SparskError) as ei:      # token outside the vocabulary: refused on the host
        P.g.decode_step_host([0], [10 ** 6], [0], [0], nt, dp)
    assert ei.value.code == binding.EINVAL
    assert [P.g.slot_state(s) for s in range(2)] == before      # nothing ran, nothing advanced
    P.g.check()
    P.close()
    # a schedule that needs a head that was not supplied
    d2 = synth.model_dims("tiny", 3, 3, 0)
    gw = binding.upload_weights(w)
    with pytest.raises(binding.SparskError) as ei:
        binding.Sparsk(d2, gw, 1, 16, 2)
    assert ei.value.code == binding.ENOHEAD


@pytest.mark.parametrize("options", [{"mega": 0}, {"mega_max_rows": 4}, {"mega_max_rows": 1, "gemm_min_rows": 2},
                                     {"mega": 0, "gemm_min_rows": 1 << 30}, {"gemm_kb": 1, "mega": 0, "gemm_min_rows": 1},
                                     {"trim_last_layer": 2}, {"trim_last_layer": 2, "mega": 0, "gemm_min_rows": 1},
                                     {"trim_last_layer": 2, "mega": 0, "gemm_min_rows": 1 << 30}, {"trim_last_layer": 0}])
def test_every_route_for_small_passes(util, options):
    """Passes of 1..4 rows (K = 4: flushes of up to three pending rows) through each of the
    implementations: the persistent kernel (also with its moving activation window at 3-4 rows),
    the tensor-core path (with 2-D descriptors too) and the small-batch kernels."""
    dims = synth.model_dims("tiny", 2, 4, 0)
    w = synth.make_weights(dims, seed=0)
    prompt = synth.make_prompts(dims, 1, 21, 21, seed=11)[0]
    P = util.Pair(dims, w, 1, 96, 3, prefill_rows=16, options=options)
    P.prefill([prompt])
    for g in range(25):
        m, c = synth.interleave(g, 1, 4)
        P.step([m], [c])
    ln, pend = P.g.slot_state(0)
    P.check_cache(0, range(1, 5), ln - pend)
    P.close()


@pytest.mark.parametrize("options", [{"attn_ctas": 2, "attn_split": 16, "mega": 0}, {"attn_ctas": 2, "attn_split": 32, "mega": 0},
                                     {"attn_ctas": 3, "attn_split": 48, "mega": 0, "attn_stages": 3},
                                     {"attn_ctas": 1, "attn_split": 64, "mega": 0, "attn_tma": 0},
                                     {"attn_ctas": 2, "attn_split": 16, "mega": 0, "attn_dynamic": 0},
                                     {"attn_ctas": 1, "mega": 0, "gemm_min_rows": 1}])
def test_attention_items_drawn_from_the_counter(util, options):
    """Many more attention work items than warps (the kernel held to one or two CTAs, four ragged
    sequences, short splits): the warps draw items from the ticket counter, launch after launch
    (the host predicts the counter's value instead of resetting it), or take every n-th item.
    Splits of one, two and three tiles with ragged ends, so that items shorter than, as long as and
    longer than a warp's ring follow one another and each starts its successor's first tiles."""
    dims = synth.model_dims("tiny", 2, 4, 0)
    w = synth.make_weights(dims, seed=0)
    prompts = synth.make_prompts(dims, 4, 9, 150, seed=21)
    P = util.Pair(dims, w, 4, 200, 3, prefill_rows=16, options=options)
    P.prefill(prompts)
    for g in range(14):
        mc = [synth.interleave(g + 2 * i, 1, 4) for i in range(4)]
        P.step([m for m, _ in mc], [c for _, c in mc])
    for s_ in range(4):
        ln, pend = P.g.slot_state(s_)
        P.check_cache(s_, range(1, 5), ln - pend)
    P.close()


@pytest.mark.parametrize("rows", [3, 10, 17, 0])
def test_prompts_share_prefill_passes(util, rows):
    """Prompts of one call are packed into passes of `rows` rows: pieces that end exactly with a pass,
    a prompt spread over several passes, several whole prompts in one, one of a single token and
    one of none; a second call appends to what the slots hold.  The cache of every layer and a
    cycle decoded on top match the oracle."""
    dims = synth.model_dims("tiny", 2, 3, 0)
    w = synth.make_weights(dims, seed=0)
    lens = [13, 2, 8, 31, 1, 6]                     # one less is ingested: the last token starts decoding
    prompts = [synth.make_prompts(dims, 1, n, n, seed=40 + i)[0] for i, n in enumerate(lens)]
    P = util.Pair(dims, w, len(lens), 64, 2, prefill_rows=rows)
    P.prefill([np.concatenate([p[:len(p) // 2], p[:1]]) for p in prompts])
    second = [p[len(p) // 2:] for p in prompts]
    P.prefill(second)
    for s_, n in enumerate(lens):
        assert P.g.slot_state(s_) == (n - 1, 0)
        if n > 1:
            P.check_cache(s_, range(1, 5), n - 1)
    for g in range(6):
        mc = [synth.interleave(g + i, 2, 4) for i in range(len(lens))]
        P.step([m for m, _ in mc], [c for _, c in mc])
    P.close()


@pytest.mark.parametrize("n", [128, 129, 300])
def test_many_prompts_in_one_prefill_pass(util, n):
    """A pass's pieces travel as kernel arguments, 128 a launch: as many, one more, and three launches over two
    passes of 256 rows; the piece behind a full launch holds several tokens."""
    dims = synth.model_dims("tiny", 2, 3, 0)
    w = synth.make_weights(dims, seed=2)
    lens = [4 if i % 64 == 0 and i else 2 for i in range(n)]
    prompts = [synth.make_prompts(dims, 1, k, k, seed=200 + i)[0] for i, k in enumerate(lens)]
    seen = sorted({0, 1, 64, 127, 128, n // 2, n - 1} & set(range(n)))
    P = util.Pair(dims, w, n, 16, 2, oracle_slots=seen)
    P.prefill(prompts)
    for s_ in seen:
        assert P.g.slot_state(s_) == (lens[s_] - 1, 0)
        P.check_cache(s_, range(1, 5), lens[s_] - 1)
    P.step([0] * n, [0] * n)
    P.close()


def test_captured_prefill_replays_and_leaves_the_context_usable(util):
    """Nothing of a prompt pass lives in host memory once it is enqueued: a captured one gives the same cache
    when it is replayed after other prompts, on tokens written to the captured buffer meanwhile, and the
    context goes on working."""
    import ctypes as C
    from paper_2603_09215_b200 import binding
    dims = synth.model_dims("tiny", 2, 3, 0)
    gw = binding.upload_weights(synth.make_weights(dims, seed=1))
    st = torch.cuda.Stream()
    st.wait_stream(torch.cuda.current_stream())
    n = 40
    prompts = [p[:n] for p in synth.make_prompts(dims, 3, n, n, seed=6)]
    with torch.cuda.stream(st):
        g = binding.Sparsk(dims, gw, 2, 64, 2, stream=st)
        tokens = torch.from_numpy(np.ascontiguousarray(prompts[0], dtype=np.int32)).cuda()
        slot, offs = (C.c_int32 * 1)(0), (C.c_int32 * 2)(0, n)
        prefill = lambda: g._check(g.lib.sparsk_prefill(g.h, 1, slot, tokens.data_ptr(), offs))
        prefill()
        st.synchronize()
        ref = []
        for p in prompts:                       # what each prompt's cache is, without a capture
            g.reset_slot(0)
            g.prefill([0], [p])
            ref.append([t.clone() for l in range(1, 5) for t in g.export_kv(0, l, 0, n)])
        g.reset_slot(0)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=st):
            prefill()
        for i in range(20):                     # more passes than any ring of staging buffers holds
            g.reset_slot(1)
            g.prefill([1], [prompts[2]])
        for i in (0, 1):
            tokens.copy_(torch.from_numpy(np.ascontiguousarray(prompts[i], dtype=np.int32)))
            graph.replay()
            got = [t for l in range(1, 5) for t in g.export_kv(0, l, 0, n)]
            st.synchronize()
            for a, b in zip(got, ref[i]):       # (the split sums' order is not fixed)
                assert float((a.float() - b.float()).abs().max()) <= 5e-3 * float(b.float().abs().max())
        g.check()
        g.close()


@pytest.mark.parametrize("B", [5, 16, 17, 64, 81, 128, 130])
def test_tcgen05_passes_of_every_width(util, B):
    """Batches on the tcgen05 path at the edges of its activation tiles (copies of 16, 32, 48 ... rows),
    on a shape whose MLP rows are dealt in units lower than the 128 rows an MMA covers."""
    dims = synth.model_dims("tiny", 2, 3, 0)
    w = synth.make_weights(dims, seed=3)
    prompts = synth.make_prompts(dims, B, 3, 12, seed=11)
    P = util.Pair(dims, w, B, 32, 2, oracle_slots=[0, B // 2, B - 1])
    P.prefill(prompts)
    for g in range(6):
        mc = [synth.interleave(g + i, 2, 4) for i in range(B)]
        P.step([m for m, _ in mc], [c for _, c in mc])
    for s_ in (0, B - 1):
        ln, pend = P.g.slot_state(s_)
        P.check_cache(s_, range(1, 5), ln - pend)
    assert P.g.route_counts()["tc"] > 0
    P.close()


@pytest.mark.parametrize("B", [5, 128])
def test_mlp_whose_gateup_units_take_two_rounds(util, B):
    """28,672 MLP rows: units of 104 rows, two for most SMs."""
    dims = synth.model_dims(dict(MICRO256, d_ffn=28672, n_layers=2), 1, 2, 0)
    w = synth.make_weights(dims, seed=17)
    prompts = synth.make_prompts(dims, B, 3, 9, seed=5)
    P = util.Pair(dims, w, B, 16, 1, oracle_slots=[0, B - 1])
    P.prefill(prompts)
    for g in range(3):
        mc = [synth.interleave(g + i, 1, 4) for i in range(B)]
        P.step([m for m, _ in mc], [c for _, c in mc])
    P.close()


@pytest.mark.parametrize("B", [9, 40, 256, 257])
@pytest.mark.parametrize("options", [{}, {"attn_split": 16, "attn_ctas": 2}])
def test_attention_of_many_ragged_sequences(util, B, options):
    """Up to 256 groups a launch numbers only the attention items with work (the longest prompt has five
    16-position splits, most have one or two), beyond that every group has as many as the longest;
    with two CTAs the items outnumber the warps many times over."""
    dims = synth.model_dims("tiny", 2, 3, 0)
    w = synth.make_weights(dims, seed=5)
    lens = [(2, 16, 17, 9, 33, 3, 48)[i % 7] for i in range(B)]
    lens[B // 2], lens[B - 1] = 70, 31
    prompts = [synth.make_prompts(dims, 1, n, n, seed=90 + i)[0] for i, n in enumerate(lens)]
    P = util.Pair(dims, w, B, 96, 2, options=dict(options, mega=0), oracle_slots=[0, 1, B // 2, B - 1])
    P.prefill(prompts)
    for g in range(4):
        mc = [synth.interleave(g + i, 2, 4) for i in range(B)]
        P.step([m for m, _ in mc], [c for _, c in mc])
    for s_ in (1, B // 2, B - 1):
        ln, pend = P.g.slot_state(s_)
        P.check_cache(s_, range(1, 5), ln - pend)
    P.close()


@pytest.mark.parametrize("options", [{}, {"attn_split": 128, "attn_ctas": 3}, {"attn_tma": 0}, {"attn_tc": 0}])
@pytest.mark.parametrize("Hq,Hkv", [(7, 1), (8, 1), (9, 1), (32, 2), (4, 2)])
def test_attention_forms_of_few_and_many_query_vectors(util, Hq, Hkv, options):
    """Head dimension 128 on the tcgen05 path: single rows of 2 to 16 query vectors per kv head, on both sides
    of the transposed item form (up to eight), and refresh blocks of four rows in blocks of 16 query vectors or,
    from 33 on, in the tcgen05 kernel (unless that is off); prefixes that end before, on and after a
    16-position tile, the 64 positions of a large block's tile and of the shortest split, and a forced
    split of 128."""
    dims = synth.model_dims(dict(MICRO256, n_layers=2, n_q_heads=Hq, n_kv_heads=Hkv, head_dim=128), 1, 4, 0)
    w = synth.make_weights(dims, seed=13)
    lens = [2, 15, 16, 17, 63, 64, 65, 128, 129, 130, 257, 390]
    prompts = [synth.make_prompts(dims, 1, n, n, seed=60 + i)[0] for i, n in enumerate(lens)]
    P = util.Pair(dims, w, len(lens), 420, 3, options=options, oracle_slots=[0, 2, 3, 5, 6, 7, 9, 11])
    P.prefill(prompts)
    for g in range(9):
        mc = [synth.interleave(g + i, 1, 4) for i in range(len(lens))]
        P.step([m for m, _ in mc], [c for _, c in mc])
    assert P.stats["max_flush"] == 3
    P.check_cache(11, range(1, 3), P.g.slot_state(11)[0] - P.g.slot_state(11)[1])
    P.close()


@pytest.mark.parametrize("n", [1, 33, 128, 129])
def test_host_and_device_buffers_give_the_same_step(util, n):
    """Up to 128 sequences a step's arrays and host tokens travel as kernel arguments, beyond that through
    staged copies; with tokens on the device the same kernels read them from there.  Slots in an
    order of their own."""
    from paper_2603_09215_b200 import binding
    dims = synth.model_dims("tiny", 2, 3, 0)
    gw = binding.upload_weights(synth.make_weights(dims, seed=6))
    prompts = synth.make_prompts(dims, n, 2, 6, seed=12)
    order = np.random.Generator(np.random.PCG64(1)).permutation(n).astype(np.int32)
    got = []
    for host in (True, False):
        g = binding.Sparsk(dims, gw, n, 16, 2)
        g.prefill(list(range(n)), [p[:-1] for p in prompts])
        tok = np.array([int(prompts[s][-1]) for s in order], np.int32)
        nt, dp = np.zeros(n, np.int32), np.zeros(n, np.int32)
        d_nt, d_dp = (torch.zeros(n, dtype=torch.int32, device="cuda") for _ in "nd")
        out = []
        for step in range(4):
            mc = [synth.interleave(step + int(s), 2, 4) for s in order]
            mods, ctrs = [m for m, _ in mc], [c for _, c in mc]
            if host:
                g.decode_step_host(order, tok, mods, ctrs, nt, dp)
            else:
                g.decode_step(order, torch.from_numpy(tok).cuda(), mods, ctrs, d_nt, d_dp)
                g.check()
                nt, dp = d_nt.cpu().numpy(), d_dp.cpu().numpy()
            out.append((nt.copy(), dp.copy()))
            tok = (tok * 7 + step) % (dims["vocab_text"] + dims["vocab_speech"])   # the same inputs on both sides
            tok = tok.astype(np.int32)
        got.append(out)
        g.close()
    for (a, da), (b, db) in zip(*got):
        assert (da == db).all()
        assert (a != b).mean() <= 0.02    # near-ties may fall either way: the split sums' order is not fixed


@pytest.mark.parametrize("shape", ["tiny", "micro64"])
@pytest.mark.parametrize("rows", [129, 161, 256, 300])
def test_prefill_passes_beyond_128_rows(util, rows, shape):
    """Products of more than 128 rows run on pairs of CTAs, each with half of the activation rows and a
    unit of weight rows of its own: odd numbers of units, rows that do not split evenly, a second
    block of rows."""
    dims = synth.model_dims("tiny" if shape == "tiny" else MICRO64, 2, 3, 0)
    w = synth.make_weights(dims, seed=4)
    prompts = synth.make_prompts(dims, 2, 150, 260, seed=8)
    P = util.Pair(dims, w, 2, 300, 2, prefill_rows=rows)
    P.prefill(prompts)
    for s_, p in enumerate(prompts):
        P.check_cache(s_, range(1, dims["n_layers"] + 1), len(p) - 1)
    P.step([0, 1], [0, 1])
    P.close()


@pytest.mark.parametrize("options", [{}, {"attn_split": 16}, {"attn_tc": 0}, {"attn_tc": 0, "attn_split": 16, "attn_tma": 0}])
def test_prefill_passes_of_several_row_blocks(util, options):
    """The library's own choice of rows a pass: a pass of 1,024 rows (four blocks of rows; attention partials have room
    for an eighth of the splits, whatever was asked for) with two groups for the tcgen05 attention and one below its
    size, then a pass with what is left."""
    dims = synth.model_dims(dict(MICRO256, n_q_heads=8, head_dim=128), 2, 3, 0)
    w = synth.make_weights(dims, seed=9)
    rng = np.random.default_rng(6)
    prompts = [rng.integers(0, 400, size=n).astype(np.int32) for n in (701, 4, 431)]
    P = util.Pair(dims, w, 3, 720, 2, options=options)
    P.prefill(prompts)
    for s_, p in enumerate(prompts):
        P.check_cache(s_, range(1, 4), len(p) - 1)
    P.step([0, 1, 0], [0, 1, 0])
    P.close()


@pytest.mark.parametrize("kb", [48, 110])
@pytest.mark.parametrize("rows", [40, 128, 256])
def test_prompt_attention_beside_small_gemm_rings(util, rows, kb):
    """Rings small enough for a GEMM CTA to share an SM with the tcgen05 attention of a prompt pass, which has
    no merge between the two: the attention takes its tensor memory before it lets the GEMM come."""
    dims = synth.model_dims(dict(MICRO256, n_q_heads=8, head_dim=128), 2, 3, 0)
    w = synth.make_weights(dims, seed=9)
    prompts = synth.make_prompts(dims, 3, 60, 300, seed=2)
    P = util.Pair(dims, w, 3, 320, 2, prefill_rows=rows, options={"gemm_smem_kb": kb}, oracle_slots=[0, 2])
    P.prefill(prompts)
    for s_ in (0, 2):
        P.check_cache(s_, range(1, 4), len(prompts[s_]) - 1)
    P.step([0, 1, 0], [0, 1, 0])
    P.close()


@pytest.mark.parametrize("d_model", [4104, 8456])
def test_wide_rows_on_the_tcgen05_path(util, d_model):
    """Residual rows wider than what the RMSNorm kernel's threads cover in one pass (4,096 numbers) and
    than what they keep in registers (8,192), not multiples of 64."""
    dims = synth.model_dims(dict(MICRO64, d_model=d_model, n_layers=2, d_ffn=96), 1, 2, 0)
    w = synth.make_weights(dims, seed=2)
    prompts = synth.make_prompts(dims, 5, 4, 9, seed=3)
    P = util.Pair(dims, w, 5, 24, 1)
    P.prefill(prompts)
    for g in range(5):
        mc = [synth.interleave(g + i, 1, 4) for i in range(5)]
        P.step([m for m, _ in mc], [c for _, c in mc])
    P.check_cache(4, range(1, 3), P.g.slot_state(4)[0] - P.g.slot_state(4)[1])
    P.close()


def test_timeout_is_reported_once_and_the_context_recovers(util):
    """A bounded in-kernel wait that runs out: the persistent kernel is told a grid-barrier count
    that no CTA can reach (a host-side test hook; nothing faults or hangs), its wait ends at the
    wall-clock limit, every CTA leaves, and the step returns SPARSK_ETIMEOUT exactly once.  The
    library then resets its barrier state by itself: after the caller resets the slot that took
    part, decoding matches the oracle again."""
    from paper_2603_09215_b200 import binding
    dims = synth.model_dims("tiny", 2, 3, 0)
    w = synth.make_weights(dims, seed=0)
    prompt = synth.make_prompts(dims, 1, 14, 14, seed=5)[0]
    P = util.Pair(dims, w, 1, 64, 2)
    P.prefill([prompt])
    for g in range(4):
        m, c = synth.interleave(g, 2, 4)
        P.step([m], [c])
    assert P.g.route_counts()["mega"] > 0                 # the steps above ran in the persistent kernel
    nt, dp = np.zeros(1, np.int32), np.zeros(1, np.int32)
    P.g.set_option("inject_barrier_timeout", 1)
    with pytest.raises(binding.SparskError) as ei:
        P.g.decode_step_host([0], [P.next_in[0]], [1], [0], nt, dp)
    assert ei.value.code == binding.ETIMEOUT
    P.g.check()                                           # reported once; the status word is clear again
    # the interrupted step left slot 0 incomplete: start it over on both sides
    P.g.reset_slot(0)
    P.os[0] = P.om.new_seq(2)
    P.g.prefill([0], [prompt[:-1]])
    P.os[0].prefill(prompt[:-1])
    P.next_in[0] = int(prompt[-1])
    for g in range(12):
        m, c = synth.interleave(g, 2, 4)
        P.step([m], [c])
    ln, pend = P.g.slot_state(0)
    P.check_cache(0, range(1, 5), ln - pend)
    P.close()


@pytest.mark.parametrize("rows", [1, 2, 4])
def test_a_ring_wait_that_runs_out_ends_the_launch_for_all(util, rows):
    """One CTA of the persistent kernel waits for bytes that do not come, in a layer that begins with the sums of the
    layer before still in their own buffer.  The other CTAs leave with it (two seconds; four where each sits out a limit of its
    own at the next barrier), and after a reset decoding matches the oracle: nothing of those sums is left."""
    import time
    from paper_2603_09215_b200 import binding
    dims = synth.model_dims(dict(MICRO256, n_layers=4), 2, 3, 0)
    w = synth.make_weights(dims, seed=0)
    prompts = [synth.make_prompts(dims, 1, 14, 14, seed=5 + i)[0] for i in range(rows)]
    P = util.Pair(dims, w, rows, 64, 2)
    P.prefill(prompts)
    P.step([0] * rows, [0] * rows)
    assert P.g.route_counts()["mega"] > 0
    nt, dp = np.zeros(rows, np.int32), np.zeros(rows, np.int32)
    P.g.set_option("inject_short_copy", 1)
    t0 = time.perf_counter()
    with pytest.raises(binding.SparskError) as ei:
        P.g.decode_step_host(list(range(rows)), P.next_in, [0] * rows, [0] * rows, nt, dp)
    took = time.perf_counter() - t0
    assert ei.value.code == binding.ETIMEOUT
    assert 1.5 < took < 3.0, took
    P.g.check()
    for s_ in range(rows):
        P.g.reset_slot(s_)
        P.os[s_] = P.om.new_seq(2)
    P.prefill(prompts)
    for g in range(7):
        mc = [synth.interleave(g, 2, 4) for _ in range(rows)]
        P.step([m for m, _ in mc], [c for _, c in mc])
    for s_ in range(rows):
        ln, pend = P.g.slot_state(s_)
        P.check_cache(s_, range(1, 5), ln - pend)
    P.close()


@pytest.mark.parametrize("options", [{}, {"mega": 0}])
@pytest.mark.parametrize("B", [2, 3])
@pytest.mark.parametrize("hd", [64, 128])
def test_partials_of_an_earlier_step_do_not_leak(util, hd, B, options):
    """A short sequence beside a long one leaves most of its attention splits empty; what their partials hold
    from an earlier step (here NaN: a cache that was imported broken, and mended afterwards) must
    not reach the output."""
    dims = synth.model_dims(dict(MICRO256, head_dim=hd), 2, 3, 0)
    w = synth.make_weights(dims, seed=29)
    lens = [300, 40, 20][:B]
    prompts = [synth.make_prompts(dims, 1, n, n, seed=70 + i)[0] for i, n in enumerate(lens)]
    P = util.Pair(dims, w, B, 330, 2, options=options)
    P.prefill(prompts)
    layers, n = range(1, dims["n_layers"] + 1), lens[0] - 1
    good = {l: tuple(t.clone() for t in P.g.export_kv(0, l, 0, n)) for l in layers}
    for l in layers:
        P.g.import_kv(0, l, 0, good[l][0], torch.full_like(good[l][1], float("nan")))
    tok, dep = np.zeros(B, np.int32), np.zeros(B, np.int32)
    for row in range(1, B):                      # the long sequence in the place of every short one
        order = list(range(B))
        order[0], order[row] = order[row], order[0]
        P.g.decode_step_host(order, np.ones(B, np.int32), [0] * B, [0] * B, tok, dep)
        for s_ in range(B):
            P.g.set_len(s_, lens[s_] - 1)
    for l in layers:
        P.g.import_kv(0, l, 0, *good[l])
    for g in range(3):
        mc = [synth.interleave(g, 1, 4)] * B
        P.step([m for m, _ in mc], [c for _, c in mc])
    P.close()


@pytest.mark.parametrize("K,maxp", [(4, 3), (3, 2)])
def test_persistent_kernel_tensor_core_form_for_three_and_four_rows(util, K, maxp):
    """Flushes of two and three pending rows (passes of three and four rows) inside the persistent
    layer-range kernel: its tensor-core form (swizzled weight boxes, mma.sync, two-term
    activations), on a shape whose inner dimensions are whole 64-element blocks."""
    dims = synth.model_dims(MICRO256, 1, K, 0)
    w = synth.make_weights(dims, seed=9)
    prompt = synth.make_prompts(dims, 1, 23, 23, seed=2)[0]
    P = util.Pair(dims, w, 1, 23 + 64, maxp, prefill_rows=16, options={"mega_max_rows": 4})
    P.prefill([prompt])
    before = P.g.route_counts()
    for g in range(30):
        m, c = synth.interleave(g, 1, K)
        P.step([m], [c])
    after = P.g.route_counts()
    assert after["tc"] == before["tc"] and after["gemv"] == before["gemv"]      # every decode pass ran in the persistent kernel
    assert P.stats["max_flush"] == K - 1
    ln, pend = P.g.slot_state(0)
    P.check_cache(0, range(1, 4), ln - pend)
    print("mega tc", P.stats)
    P.close()


@pytest.mark.parametrize("rows", [3, 4])
@pytest.mark.parametrize("d_ffn", [4352, 9280, 18944, 18976 + 32])
def test_persistent_kernel_mlp_shares(util, rows, d_ffn):
    """Three and four rows in the persistent kernel with an MLP of which a CTA has one box of 128 columns at most, filled
    to the last, and just more, which takes the wide form (148 SMs)."""
    dims = synth.model_dims(dict(MICRO256, d_ffn=d_ffn, n_layers=2), 1, 4, 0)
    w = synth.make_weights(dims, seed=19)
    prompts = synth.make_prompts(dims, rows, 5, 30, seed=4)
    P = util.Pair(dims, w, rows, 64, 3)
    P.prefill(prompts)
    before = P.g.route_counts()["mega"]
    for g in range(5):
        mc = [synth.interleave(g, 1, 4)] * rows
        P.step([m for m, _ in mc], [c for _, c in mc])
    assert P.g.route_counts()["mega"] > before
    P.check_cache(rows - 1, range(1, 3), P.g.slot_state(rows - 1)[0] - P.g.slot_state(rows - 1)[1])
    P.close()


@pytest.mark.parametrize("d_model,route", [(4352, "mega"), (4416, "tc"), (5120, "tc")])
@pytest.mark.parametrize("rows", [1, 3, 4])
def test_three_and_four_wide_rows(util, rows, d_model, route):
    """Residual rows that just fit the persistent kernel's activation area as three or four rows, and rows
    that do not, which take the tcgen05 path: batches of three and four, and one sequence whose
    refresh carries three pending rows."""
    dims = synth.model_dims(dict(MICRO256, d_model=d_model, n_layers=2, d_ffn=128), 1, 4, 0)
    w = synth.make_weights(dims, seed=23)
    prompts = synth.make_prompts(dims, rows, 5, 20, seed=7)
    P = util.Pair(dims, w, rows, 64, 3)
    P.prefill(prompts)
    other = "tc" if route == "mega" else "mega"
    for g in range(6):
        before = P.g.route_counts()
        P.step([0 if g == 0 else 1] * rows, [0 if g == 0 else g - 1] * rows)
        after = P.g.route_counts()
        if rows >= 3 or g == 5:              # g = 5 is the refresh: three pending rows and the current one
            assert after[route] > before[route]
        if (rows >= 3 and g < 5) or (rows == 1 and route == "mega"):
            assert after[other] == before[other]
    assert P.stats["max_flush"] == 3
    P.check_cache(rows - 1, range(1, 3), P.g.slot_state(rows - 1)[0] - P.g.slot_state(rows - 1)[1])
    P.close()


@pytest.mark.parametrize("shape,lens", [
    # a CTA's MLP columns: none for most CTAs, a lone band, boxes that reach into the next CTA's columns
    (dict(d_model=256, n_q_heads=4, n_kv_heads=2, head_dim=64, d_ffn=64), (1,)),
    (dict(d_model=200, n_q_heads=6, n_kv_heads=3, head_dim=64, d_ffn=712), (17, 30)),
    # 148 SMs x 128 columns and a little: the wide form; nine bands a CTA meet in two batches of sums
    (dict(d_model=64, n_q_heads=2, n_kv_heads=1, head_dim=128, d_ffn=19200), (33,)),
    (dict(d_model=128, n_q_heads=2, n_kv_heads=2, head_dim=64, d_ffn=19008), (5, 64, 16)),
    # sixteen query heads a kv head (two blocks of eight query vectors), fewer cache tiles than SMs; three or four tiles a CTA
    (dict(d_model=192, n_q_heads=16, n_kv_heads=1, head_dim=64, d_ffn=320), (900, 3)),
    (dict(d_model=128, n_q_heads=8, n_kv_heads=4, head_dim=64, d_ffn=256), (1300, 15, 48, 700)),
    # wide form with a last block of 128 columns that is ragged, one to four rows
    (dict(d_model=136, n_q_heads=2, n_kv_heads=1, head_dim=128, d_ffn=19016), (21,)),
    (dict(d_model=136, n_q_heads=2, n_kv_heads=1, head_dim=64, d_ffn=19016), (21, 5)),
    (dict(d_model=192, n_q_heads=2, n_kv_heads=2, head_dim=128, d_ffn=38080), (21, 5, 30, 12)),
    # a residual row wider than the registers of the norm hold; one that needs the wide form, just not and just so; whole with one row
    # and two rows, and in windows
    (dict(d_model=4352, n_q_heads=2, n_kv_heads=1, head_dim=64, d_ffn=128), (20,)),
    (dict(d_model=7168, n_q_heads=2, n_kv_heads=1, head_dim=64, d_ffn=2400), (20,)),
    (dict(d_model=7176, n_q_heads=2, n_kv_heads=1, head_dim=128, d_ffn=2400), (20,)),
    (dict(d_model=11264, n_q_heads=2, n_kv_heads=1, head_dim=64, d_ffn=64), (18, 9)),
    (dict(d_model=11520, n_q_heads=2, n_kv_heads=1, head_dim=64, d_ffn=256), (18, 9)),
    (dict(d_model=23808, n_q_heads=2, n_kv_heads=1, head_dim=64, d_ffn=2400), (18,)),
])
def test_persistent_kernel_at_the_edges_of_its_shares(util, shape, lens):
    """One to four rows through the persistent kernel (and the flushes of what they leave pending where those are
    as few) where the shares of its CTAs are empty, ragged, or more than one box, run or window."""
    dims = synth.model_dims(dict(n_layers=3, vocab_text=96, vocab_speech=64, rms_eps=1e-6, rope_base=10000.0, **shape), 2, 3, 0)
    w = synth.make_weights(dims, seed=3)
    rng = np.random.default_rng(5)
    prompts = [rng.integers(0, 160, size=n + 1).astype(np.int32) for n in lens]
    P = util.Pair(dims, w, len(lens), max(lens) + 16, 2, prefill_rows=64)
    P.prefill(prompts)
    before = P.g.route_counts()["mega"]
    for g in range(7):
        mc = [synth.interleave(g + i, 1, 4) for i in range(len(lens))]
        P.step([m for m, _ in mc], [c for _, c in mc])
    assert P.g.route_counts()["mega"] > before
    for s_ in range(len(lens)):
        ln, pend = P.g.slot_state(s_)
        P.check_cache(s_, range(1, 4), ln - pend)
    P.close()


@pytest.mark.parametrize("hd,n_kv,G,lens", [
    # shares of five and six tiles (16 positions of a kv head) on 148 SMs: runs of one share side by side, two warps a run
    (64, 16, 1, (760,)), (128, 16, 1, (900,)),
    # of ten: three warps with twelve slots, two with eight; a share's runs have more tiles than the ring
    (64, 16, 2, (1480,)), (128, 8, 4, (600, 700, 800, 900)), (64, 16, 2, (400, 1100)),
    # of 34: a run goes round the ring more than once; of seventeen, four rows of four blocks of query vectors
    (128, 16, 1, (5100,)), (64, 16, 2, (1300, 1290, 1280, 1310)), (64, 8, 8, (5100,)),
    # more query vectors a group than a warp a block of eight takes in one go
    (64, 1, 64, (3000,)), (64, 1, 72, (900, 2000)), (128, 1, 40, (12000,)),
])
def test_persistent_kernel_long_runs(util, hd, n_kv, G, lens):
    """Attention of the persistent kernel where a CTA's share of the cache is long, over imported prefixes: one to four
    sequences, and the refresh passes of what they leave pending."""
    dims = synth.model_dims(dict(n_layers=2, d_model=64, n_q_heads=n_kv * G, n_kv_heads=n_kv, head_dim=hd, d_ffn=128, vocab_text=96,
                                 vocab_speech=64, rms_eps=1e-6, rope_base=10000.0), 1, 4, 0)
    P = util.Pair(dims, synth.make_weights(dims, seed=3), len(lens), max(lens) + 16, 3, prefill_rows=64)
    rng = np.random.default_rng(8)
    for s_, n in enumerate(lens):
        for layer in (1, 2):
            k, v = (rng.standard_normal((n, n_kv * hd)).astype(np.float16) for _ in "kv")
            P.g.import_kv(s_, layer, 0, torch.from_numpy(k).cuda(), torch.from_numpy(v).cuda())
            kf, vf = k.astype(np.float64), v.astype(np.float64)
            for p in range(n):
                P.os[s_].set_kv(layer, p, kf[p], vf[p])
        P.g.set_len(s_, n)
        P.os[s_].set_len(n)
    P.next_in = [int(t) for t in rng.integers(0, 160, size=len(lens))]
    for g in range(6):
        before = P.g.route_counts()
        P.step([0 if g == 0 else 1] * len(lens), [0 if g == 0 else g - 1] * len(lens))
        after = P.g.route_counts()
        if g < 5 or len(lens) == 1:              # g = 5 is the refresh: three pending rows a sequence
            assert after["mega"] > before["mega"] and after["tc"] == before["tc"] and after["gemv"] == before["gemv"]
    assert P.stats["max_flush"] == 3
    P.close()


@pytest.mark.parametrize("lens,passes", [((256,), 1), ((257,), 2), ((288,), 2), ((289,), 1), ((230, 40), 2), ((300, 229), 1), ((512, 100, 200), 1),
                                         ((1030,), 2)])
def test_prompt_rows_behind_whole_blocks(util, lens, passes):
    """The library's own choice of rows a pass: few rows behind whole blocks of 256 go by themselves where their block would need
    another wave of gate/up units (38 pairs of them on 74 pairs of SMs), the next prompt's rows with them."""
    dims = synth.model_dims(dict(MICRO256, n_layers=2, d_ffn=9728), 1, 3, 0)
    P = util.Pair(dims, synth.make_weights(dims, seed=9), len(lens), max(lens) + 4, 2)
    rng = np.random.default_rng(6)
    prompts = [rng.integers(0, 400, size=n + 1).astype(np.int32) for n in lens]
    P.prefill(prompts)
    assert sum(P.g.route_counts().values()) == 2 * passes
    for s_, n in enumerate(lens):
        P.check_cache(s_, (1, 2), n)
    P.step([0] * len(lens), [0] * len(lens))
    P.close()


@pytest.mark.parametrize("hd,G,short,n,passes", [
    (64, 2, 2, 4000, 1), (64, 2, 40, 4000, 1), (128, 2, 2, 4000, 1), (128, 2, 40, 4000, 1), (128, 8, 2, 4000, 1), (128, 8, 40, 4000, 1),
    (128, 2, 2, 30000, 2),
])
def test_few_prompt_rows_behind_a_long_prefix(util, hd, G, short, n, passes):
    """A prompt pass whose groups are uneven (few rows behind n positions beside many rows of a new prompt) takes more splits
    than the largest group alone would have, in either attention kernel and in both at once; where a pass of all rows has no
    room for enough of them it has 256 of them."""
    dims = synth.model_dims(dict(n_layers=2, d_model=64, n_q_heads=8 * G, n_kv_heads=8, head_dim=hd, d_ffn=128, vocab_text=96,
                                 vocab_speech=64, rms_eps=1e-6, rope_base=10000.0), 1, 4, 0)
    rng = np.random.default_rng(12)
    P = util.Pair(dims, synth.make_weights(dims, seed=3), 2, n + 64, 3)
    for layer in (1, 2):
        k, v = (rng.standard_normal((n, 8 * hd)).astype(np.float16) for _ in "kv")
        P.g.import_kv(0, layer, 0, torch.from_numpy(k).cuda(), torch.from_numpy(v).cuda())
        kf, vf = k.astype(np.float64), v.astype(np.float64)
        for p in range(n):
            P.os[0].set_kv(layer, p, kf[p], vf[p])
    P.g.set_len(0, n)
    P.os[0].set_len(n)
    P.prefill([rng.integers(0, 160, size=m + 1).astype(np.int32) for m in (short, 600)])
    assert sum(P.g.route_counts().values()) == 2 * passes
    P.check_cache(0, (1, 2), n + short)
    P.check_cache(1, (1, 2), 600)
    P.step([0, 0], [0, 0])
    P.close()
