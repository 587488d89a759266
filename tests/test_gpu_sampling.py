"""GPU parity of nucleus sampling (Sec. V-A: temperature 0.7, top_p 0.9) against the reference
sampler.  The two sides sum the same probabilities in different orders and precisions, so a token
is accepted when the uniform number lies inside, or within LAND_TOL of, the cumulative interval
the reference order gives that token (intervals of a flat 150k-id distribution are ~1e-5 wide, so
exact equality is only demanded where the reference's own landing point is well inside)."""
import numpy as np
import pytest
import torch

from paper_2603_09215_b200 import synth

pytestmark = pytest.mark.gpu

T, TOP_P = 0.7, 0.9
LAND_TOL = 3e-5     # fp32 sums of up to 152k weights against float64 (n * 2^-24 / sqrt-ish growth, with margin)


@pytest.fixture(scope="module")
def mods():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from oracle import sampling as smp
    from paper_2603_09215_b200 import binding
    return smp, binding


def _run(binding, z, u, modality, Vt, Vs, temperature=T, top_p=TOP_P):
    zt = torch.from_numpy(z).cuda()
    ut = torch.from_numpy(np.asarray(u, np.float32)).cuda()
    mt = torch.tensor(modality, dtype=torch.int32, device="cuda")
    out = binding.nucleus_sample(zt, ut, mt, Vt, Vs, temperature, top_p)
    torch.cuda.synchronize()
    return out.cpu().numpy()


@pytest.mark.parametrize("Vt,Vs,scale,seed", [(1024, 512, 0.3, 1), (151936, 6561, 1.2, 2), (151552, 16384, 0.3, 3),
                                              (301, 99, 4.0, 4), (5000, 1, 1.0, 5), (1000, 0, 8.0, 6)])
def test_tokens_land_where_the_reference_puts_them(mods, Vt, Vs, scale, seed):
    smp, binding = mods
    n = 24
    z = synth.make_logits(n, Vt + Vs, scale, seed)
    u = synth.make_uniforms(n, seed + 100)
    modality = [(i % 3 != 0) and Vs > 0 for i in range(n)]
    got = _run(binding, z, u, [int(m) for m in modality], Vt, Vs)
    exact = 0
    for i in range(n):
        lo, hi = (Vt, Vt + Vs) if modality[i] else (0, Vt)
        ref = smp.nucleus_sample(z[i], lo, hi, T, TOP_P, float(u[i]))
        assert lo <= got[i] < hi
        err = smp.landing_error(ref, int(got[i]), float(u[i]))
        assert err <= LAND_TOL, (i, int(got[i]), ref["token"], err)
        exact += int(got[i]) == ref["token"]
        # where the reference's landing point is well inside its interval the token is the same one
        j = ref["rank"]
        inside = min(float(u[i]) - (ref["cum"][j - 1] if j else 0.0), ref["cum"][j] - float(u[i]))
        if inside > 4 * LAND_TOL:
            assert int(got[i]) == ref["token"], (i, inside)
    print("exact", exact, "of", n)


@pytest.mark.parametrize("Vt,Vs", [(8192, 8193), (24576, 24577), (511, 513), (8191, 31)])
def test_ranges_at_the_ends_of_the_kernel_forms(mods, Vt, Vs):
    """16 weights a thread up to 8,192 ids, 48 up to 24,576, a cluster beyond; ranges that leave threads without ids."""
    smp, binding = mods
    n = 12
    z = synth.make_logits(n, Vt + Vs, 1.0, Vt)
    z[::4, 1::2] = z[::4, 0:1]  # some rows with half of their ids tied
    u = synth.make_uniforms(n, Vs)
    got = _run(binding, z, u, [i % 2 for i in range(n)], Vt, Vs)
    for i in range(n):
        lo, hi = (Vt, Vt + Vs) if i % 2 else (0, Vt)
        ref = smp.nucleus_sample(z[i], lo, hi, T, TOP_P, float(u[i]))
        assert lo <= got[i] < hi
        assert smp.landing_error(ref, int(got[i]), float(u[i])) <= LAND_TOL, (i, int(got[i]), ref["token"])


def test_worked_example_limits_and_ties(mods):
    smp, binding = mods
    z = np.log(np.array([[0.05, 0.5, 0.15, 0.3]] * 4, dtype=np.float32))
    assert list(_run(binding, z, [0.5, 0.6, 0.9, 0.999], [0] * 4, 4, 0, 1.0, 0.9)) == [1, 3, 2, 2]
    assert list(_run(binding, z, [0.7, 0.8, 0.0, 0.99], [0] * 4, 4, 0, 0.5, 0.9)) == [1, 3, 1, 3]
    # limits that reduce to the arg max: a vanishing nucleus, a vanishing temperature
    zz = synth.make_logits(6, 700, 1.0, 9)
    u = [0.0, 0.2, 0.5, 0.7, 0.9, 0.999]
    best = zz[:, :500].argmax(1)
    assert list(_run(binding, zz, u, [0] * 6, 500, 200, 0.7, 1e-9)) == list(best)
    assert list(_run(binding, zz, u, [0] * 6, 500, 200, 1e-4, 0.9)) == list(best)
    assert list(_run(binding, zz, u, [1] * 6, 500, 200, 0.7, 1e-9)) == list(500 + zz[:, 500:].argmax(1))
    # equal logits: ids in order, top_p = 1 keeps them all
    flat = np.zeros((4, 10), np.float32)
    assert list(_run(binding, flat, [0.0, 0.17, 0.55, 0.99], [1] * 4, 2, 8, 0.7, 1.0)) == [2, 3, 6, 9]
    # the logits are only read
    z2 = synth.make_logits(3, 900, 2.0, 10)
    zt = torch.from_numpy(z2).cuda()
    binding.nucleus_sample(zt, torch.tensor([0.1, 0.5, 0.9], device="cuda"), torch.tensor([0, 1, 0], dtype=torch.int32, device="cuda"),
                           600, 300, T, TOP_P)
    torch.cuda.synchronize()
    assert np.array_equal(zt.cpu().numpy(), z2)
    # a range larger than one cluster holds is refused
    with pytest.raises(binding.SparskError):
        binding.nucleus_sample(torch.zeros((1, 200000), device="cuda"), torch.zeros(1, device="cuda"),
                               torch.zeros(1, dtype=torch.int32, device="cuda"), 200000, 0, T, TOP_P)


def test_bad_arguments_are_refused(mods):
    smp, binding = mods
    z = torch.zeros((2, 8), dtype=torch.float32, device="cuda")
    u = torch.zeros(2, dtype=torch.float32, device="cuda")
    m = torch.zeros(2, dtype=torch.int32, device="cuda")
    for temperature, top_p in ((0.0, 0.9), (-1.0, 0.9), (float("inf"), 0.9), (0.7, 0.0), (0.7, 1.5), (float("nan"), 0.9)):
        with pytest.raises(binding.SparskError):
            binding.nucleus_sample(z, u, m, 8, 0, temperature, top_p)


def test_decode_steps_with_sampling_follow_the_reference(mods):
    """The whole step with sampling switched on: depths bit-exact, and every token lands where the
    reference sampler, run on the ORACLE's logits with the same uniform number, puts it, within a
    tolerance for the 2e-2 the logits may differ by; both sides continue on the reference token."""
    smp, binding = mods
    from oracle import oracle as ora
    dims = synth.model_dims("tiny", 2, 3, 0)
    w = synth.make_weights(dims, seed=0)
    B, steps = 3, 30
    prompts = synth.make_prompts(dims, B, 10, 24, seed=5)
    g = binding.Sparsk(dims, binding.upload_weights(w), B, 24 + steps + 1, 2, 16)
    om = ora.OracleModel(dims, w, max_len=24 + steps + 1)
    seqs = [om.new_seq(2) for _ in range(B)]
    g.prefill(list(range(B)), [p[:-1] for p in prompts])
    for s, p in zip(seqs, prompts):
        s.prefill(p[:-1])
    nxt = [int(p[-1]) for p in prompts]
    uni = torch.zeros(B, dtype=torch.float32, device="cuda")
    g.set_sampling(T, TOP_P, uni)
    tok = torch.zeros(B, dtype=torch.int32, device="cuda")
    out_t = torch.zeros(B, dtype=torch.int32, device="cuda")
    out_d = torch.zeros(B, dtype=torch.int32, device="cuda")
    Vt, V = dims["vocab_text"], dims["vocab_text"] + dims["vocab_speech"]
    phases = [0, 2, 5]
    exact, worst = 0, 0.0
    for st in range(steps):
        mc = [synth.interleave(st, 2, 4, ph) for ph in phases]
        u = synth.make_uniforms(B, 1000 + st)
        uni.copy_(torch.from_numpy(u))
        tok.copy_(torch.tensor(nxt, dtype=torch.int32))
        g.decode_step(list(range(B)), tok, [m for m, _ in mc], [c for _, c in mc], out_t, out_d)
        g.check()
        got_t, got_d = out_t.cpu().numpy(), out_d.cpu().numpy()
        for b in range(B):
            m, c = mc[b]
            r = seqs[b].decode_step(nxt[b], m, c)
            assert got_d[b] == r["depth"]
            lo, hi = (0, Vt) if m == 0 else (Vt, V)
            ref = smp.nucleus_sample(r["logits"], lo, hi, T, TOP_P, float(u[b]))
            err = smp.landing_error(ref, int(got_t[b]), float(u[b]))
            assert err <= 2e-2, (st, b, int(got_t[b]), ref["token"], err)
            worst = max(worst, err)
            exact += int(got_t[b]) == ref["token"]
            nxt[b] = ref["token"]
    print("sampling steps: exact", exact, "of", steps * B, "worst landing error", worst)
    assert exact > steps * B // 2
    # back to greedy decoding
    g.set_sampling(0, 1, None)
    tok.copy_(torch.tensor(nxt, dtype=torch.int32))
    g.decode_step(list(range(B)), tok, [1] * B, [0] * B, out_t, out_d)
    g.check()
    for b in range(B):
        r = seqs[b].decode_step(nxt[b], 1, 0)
        if r["margin"] > 5e-2:
            assert int(out_t.cpu()[b]) == r["token"]
    g.close()
