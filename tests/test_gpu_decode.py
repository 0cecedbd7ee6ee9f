"""GPU parity of the decode entry points and the cache append against the CPU oracle."""
import dataclasses

import numpy as np
import pytest
import torch

import oracle
from paper_2408_01890_b200 import binding as lb
from paper_2408_01890_b200 import synth
from helpers import ACT, assert_close, dev, f64

pytestmark = pytest.mark.gpu


def fill_shared_cache(w, t, B, L, L_cap, dtype):
    cache = lb.KVCacheLayer(lb.CACHE_SHARED, B, w.Hkv, L_cap, w.d, w.r, dtype=dtype)
    lb.lisa_kvcache_append(cache, dev(t["kp"]), dev(t["v"]))
    return cache


def run_shared_decode(w, B, L, lens=None, seed=0, integrate=lb.INTEGRATE_ADD, ffn_layers=2, bias=False, L_cap=None):
    tdt = torch.bfloat16 if w.dtype == "bf16" else torch.float32
    L_cap = L_cap or ((L + 7) // 8 * 8)
    t = synth.decode_inputs(w, seed, B=B, L=L)
    m = w.Hq if ffn_layers == 1 else w.m
    hin = 2 * w.Hq if integrate == lb.INTEGRATE_CONCAT else w.Hq
    w1 = synth.as_dtype(synth.normal("w1", (hin, m), seed, std=hin ** -0.5), w.dtype)
    w2 = synth.as_dtype(synth.normal("w2", (m, w.Hq), seed, std=m ** -0.5), w.dtype) if ffn_layers == 2 else None
    b1 = synth.as_dtype(synth.normal("b1", (m,), seed, std=0.5), w.dtype) if bias else None
    b2 = synth.as_dtype(synth.normal("b2", (w.Hq,), seed, std=0.5), w.dtype) if (bias and ffn_layers == 2) else None
    cache = fill_shared_cache(w, t, B, L, L_cap, tdt)
    lens_h = np.full((B,), L, dtype=np.int32) if lens is None else np.asarray(lens, dtype=np.int32)
    lens_d = None if lens is None else torch.from_numpy(lens_h).cuda()
    link = lb.Link(dev(t["qp"]), None, dev(w1), None if w2 is None else dev(w2), None if b1 is None else dev(b1),
                   None if b2 is None else dev(b2), act=ACT[w.act][0], integrate=integrate, ffn_layers=ffn_layers)
    row = torch.full((B, w.Hq, L_cap), -7.0, dtype=torch.float32, device="cuda")
    out = lb.lisa_attn_shared_decode(dev(t["prev"]), link, cache, L=L, seq_lens=lens_d, out_scores=row)
    out_norow = lb.lisa_attn_shared_decode(dev(t["prev"]), link, cache, L=L, seq_lens=lens_d)
    torch.cuda.synchronize()
    olink = oracle.Link(None, None, f64(w1), f64(w2), f64(b1), f64(b2), r=w.r, act=ACT[w.act][1], integrate=integrate,
                        ffn_layers=ffn_layers)
    O, R = oracle.decode_shared(f64(t["prev"]), f64(t["qp"])[:, 0], f64(t["kp"]), f64(t["v"]), olink, lens_h)
    assert_close(out[:, 0].float().cpu().numpy(), O, w.dtype, "decode O")
    assert torch.equal(out, out_norow)
    row_h = row.cpu().numpy()
    for b in range(B):
        assert_close(row_h[b, :, :lens_h[b]], R[b, :, :lens_h[b]], "f32" if w.dtype == "f32" else "bf16", "score row")
        assert np.all(row_h[b, :, lens_h[b]:] == -7.0), "row written beyond the sequence length"
    assert lb.lisa_check() == lb.OK


D_SMALL = synth.Workload("dsmall", "bf16", 3, 300, 8, 2, 64, 21, 16, "relu", 1, True)


@pytest.mark.parametrize("integrate,act,layers,bias", [
    (lb.INTEGRATE_ADD, "relu", 2, False), (lb.INTEGRATE_ADD, "silu", 2, True), (lb.INTEGRATE_CONCAT, "relu", 2, True),
    (lb.INTEGRATE_CONCAT, "none", 1, False), (lb.INTEGRATE_PLUS, "none", 2, False)])
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_shared_decode_modes(integrate, act, layers, bias, dtype):
    w = dataclasses.replace(D_SMALL, dtype=dtype, act=act)
    run_shared_decode(w, 3, 300, lens=[300, 1, 129], seed=2, integrate=integrate, ffn_layers=layers, bias=bias)


@pytest.mark.parametrize("Hq,Hkv,d,r,m,L", [(40, 40, 128, 21, 80, 700), (32, 32, 128, 21, 64, 515), (32, 8, 128, 20, 64, 260),
                                              (4, 4, 32, 8, 16, 128), (3, 1, 32, 1, 6, 9)])
def test_shared_decode_shapes(Hq, Hkv, d, r, m, L):
    w = synth.Workload("dshape", "bf16", 2, L, Hq, Hkv, d, r, m, "relu", 1, True)
    run_shared_decode(w, 2, L, lens=[L, max(1, L // 3)], seed=4)
    run_shared_decode(w, 2, L, lens=None, seed=5, L_cap=(L + 7) // 8 * 8 + 64)


def sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


@pytest.mark.parametrize("Hq,Hkv,m,B,L", [(32, 8, 64, 10, 4200), (40, 40, 80, 12, 3500), (32, 32, 64, 50, 385)])
def test_shared_decode_three_ctas_per_sm(Hq, Hkv, m, B, L):
    """Grids of 297..444 chunk CTAs (on 148 SMs) take the build of the chunk kernel that runs three CTAs per SM: all sequences of the
    call's length (by grid coordinates; the last chunk is partial), then ragged lengths (dealt), against the oracle like every other shape.
    The last shape runs with sixteen heads to a CTA."""
    w = synth.Workload("dthree", "bf16", B, L, Hq, Hkv, 128, 21, m, "relu", 1, True)
    run_shared_decode(w, B, L, lens=None, seed=5)
    lens = [L if b % 3 == 0 else (1 + (b * 977) % L) for b in range(B)]
    run_shared_decode(w, B, L, lens=lens, seed=6)


@pytest.mark.parametrize("per_sm,L", [(8, 1100), (10, 1100), (10, 700)])
def test_merges_of_grids_around_the_resident_ones(per_sm, L):
    """The merge holds eight, two or one partial outputs of a thread ahead, by how many of its CTAs an SM holds: batches just beyond eight
    and ten CTAs per SM, with more chunks than are held ahead and sequences of every number of chunks."""
    B = per_sm * sms() // 32 + 1
    w = synth.Workload("dmerge", "bf16", B, L, 32, 8, 128, 21, 64, "relu", 1, True)
    run_shared_decode(w, B, L, lens=[max(1, L * (b + 1) // B) for b in range(B)], seed=11)


@pytest.mark.parametrize("Hq,Hkv,m,L", [(32, 8, 64, 3201), (40, 40, 80, 2625)])
@pytest.mark.parametrize("more", ["all", 1, 0])
def test_the_count_of_a_dealt_batch_picks_its_build(Hq, Hkv, m, L, more):
    """Given lengths, a grid of two to three CTAs per SM: with one chunk that holds positions more than two per SM, up to all of them, the
    build for three per SM does the work, with no more than two per SM the other.  Both are launched (and the merge): lengths are on the device."""
    nc, slots = (L + 127) // 128, 2 * sms()
    B = slots // nc + 2
    assert slots < B * nc <= 3 * sms() and B <= 32
    if more == "all":
        lens = [L] * B
    else:   # every sequence keeps a chunk; the first ones give up whole chunks until slots + more are left
        spare, lens = B * nc - slots - more, []
        for b in range(B):
            cut = min(spare, nc - 1)
            spare -= cut
            lens.append(L - 128 * cut)
        assert sum((x + 127) // 128 for x in lens) == slots + more and min(lens) >= 1
    w = synth.Workload("dpair", "bf16", B, L, Hq, Hkv, 128, 21, m, "relu", 1, True)
    n0 = lb.lisa_kernel_launches()
    run_shared_decode(w, B, L, lens=lens, seed=7)
    assert lb.lisa_kernel_launches() - n0 == 1 + 2 * 3   # the append, two calls


@pytest.mark.parametrize("Hq,Hkv,m,act,integrate,B,L", [
    (32, 32, 64, "relu", lb.INTEGRATE_ADD, 1, 31), (32, 16, 64, "silu", lb.INTEGRATE_ADD, 2, 33), (40, 40, 80, "relu", lb.INTEGRATE_ADD, 3, 65),
    (32, 4, 64, "relu", lb.INTEGRATE_ADD, 1, 1000),          # eight query heads to a KV head, chunks of 32 and 64 positions
    (32, 8, 64, "relu", lb.INTEGRATE_ADD, 9, 1100),          # heads in groups, chunks of 128
    (32, 32, 64, "relu", lb.INTEGRATE_ADD, 50, 385),         # sixteen heads to a CTA
    (32, 32, 256, "relu", lb.INTEGRATE_CONCAT, 2, 257), (32, 8, 72, "silu", lb.INTEGRATE_CONCAT, 30, 640), (40, 8, 128, "relu", lb.INTEGRATE_CONCAT, 2, 130),
    (32, 8, 256, "relu", lb.INTEGRATE_ADD, 1, 97), (40, 40, 24, "silu", lb.INTEGRATE_ADD, 3, 700)])
def test_shared_decode_small_and_grouped(Hq, Hkv, m, act, integrate, B, L):
    """Every way a launch is cut: chunk lengths, groups of heads, query heads that share a KV head, FFN widths off the compiled ones."""
    w = synth.Workload("dcut", "bf16", B, L, Hq, Hkv, 128, 21, m, act, 1, True)
    lens = [max(1, (L * (b + 1)) // B - b % 3) for b in range(B)]
    run_shared_decode(w, B, L, lens=lens, seed=8, integrate=integrate, bias=True)


@pytest.mark.parametrize("Hq,Hkv,B,L", [(32, 32, 1, 31), (32, 16, 2, 65), (32, 8, 3, 129), (32, 4, 20, 1030), (40, 8, 2, 300), (2, 1, 1, 17)])
def test_anchor_decode_cuts(Hq, Hkv, B, L):
    """The standard layer's chunk lengths, groups of KV heads and shared KV heads, sequences that end inside a chunk."""
    w = synth.Workload("acut", "bf16", B, L, Hq, Hkv, 128, 8, 16, "relu", 1, True)
    t = synth.decode_inputs(w, 7, B=B, L=L)
    cache = lb.KVCacheLayer(lb.CACHE_STANDARD, B, Hkv, (L + 7) // 8 * 8, 128)
    lb.lisa_kvcache_append(cache, dev(t["k"]), dev(t["v"]))
    lens = np.array([max(1, (L * (b + 1)) // B - b % 3) for b in range(B)], dtype=np.int32)
    row = torch.full((B, Hq, cache.L_cap), -7.0, dtype=torch.float32, device="cuda")
    out = lb.lisa_attn_anchor(dev(t["q0"]), cache=cache, L=L, seq_lens=torch.from_numpy(lens).cuda(), out_scores=row)
    O, R = oracle.decode_anchor(f64(t["q0"])[:, 0], f64(t["k"]), f64(t["v"]), lens)
    assert_close(out[:, 0].float().cpu().numpy(), O, "bf16", "anchor decode O")
    row_h = row.cpu().numpy()
    for b in range(B):
        assert_close(row_h[b, :, :lens[b]], R[b, :, :lens[b]], "f32", "anchor score row")
        assert np.all(row_h[b, :, lens[b]:] == -7.0)


@pytest.mark.parametrize("Hq,Hkv,L", [(32, 32, 333), (32, 16, 45), (32, 8, 1111), (40, 40, 7)])
def test_an_infinity_in_the_last_row_stays_one(Hq, Hkv, L):
    """A sequence that ends inside a chunk, its last V row holding an infinity: that column of the output is infinite, as softmax times V
    is, and no other column is touched."""
    w = synth.Workload("inf", "bf16", 1, L, Hq, Hkv, 128, 21, 2 * Hq, "relu", 1, True)
    t = synth.decode_inputs(w, 9, B=1, L=L)
    clean = t["v"].clone()
    t["v"][0, L - 1, :, 5] = float("inf")
    L_cap = (L + 7) // 8 * 8
    shared = fill_shared_cache(w, t, 1, L, L_cap, torch.bfloat16)
    standard = lb.KVCacheLayer(lb.CACHE_STANDARD, 1, Hkv, L_cap, 128)
    lb.lisa_kvcache_append(standard, dev(t["k"]), dev(t["v"]))
    got = [lb.lisa_attn_shared_decode(dev(t["prev"]), lb.Link(dev(t["qp"]), None, dev(t["w1"]), dev(t["w2"])), shared, L=L),
           lb.lisa_attn_anchor(dev(t["q0"]), cache=standard, L=L)]
    olink = oracle.Link(None, None, f64(t["w1"]), f64(t["w2"]), r=w.r, act=ACT["relu"][1])
    lens = np.array([L], dtype=np.int32)
    ref = [oracle.decode_shared(f64(t["prev"]), f64(t["qp"])[:, 0], f64(t["kp"]), f64(clean), olink, lens)[0],
           oracle.decode_anchor(f64(t["q0"])[:, 0], f64(t["k"]), f64(clean), lens)[0]]
    others = [x for x in range(128) if x != 5]
    for o, r in zip(got, ref):
        o = o[:, 0].float().cpu().numpy()
        assert np.all(np.isposinf(o[:, :, 5]))
        assert_close(o[:, :, others], r[:, :, others], "bf16", "columns without an infinity")


@pytest.mark.parametrize("Hq,m,integrate", [(32, 256, lb.INTEGRATE_CONCAT), (32, 72, lb.INTEGRATE_ADD), (40, 24, lb.INTEGRATE_ADD)])
def test_the_lowest_score_stays_finite(Hq, m, integrate):
    """Previous scores of the type's lowest value at some positions, through an FFN whose weights keep its sums below the type's largest:
    results stay finite and are the oracle's, as with any other scores."""
    B, L = 2, 77
    w = synth.Workload("lowest", "bf16", B, L, Hq, Hq, 128, 21, m, "relu", 1, True)
    t = synth.decode_inputs(w, 10, B=B, L=L)
    at = [3, 40, 76]
    t["prev"][:, :, at] = torch.finfo(torch.float32).min
    h_in = Hq * (2 if integrate == lb.INTEGRATE_CONCAT else 1)
    w1 = synth.as_dtype(synth.normal("w1", (h_in, m), 10, std=0.02), "bf16")
    w2 = synth.as_dtype(synth.normal("w2", (m, Hq), 10, std=0.02), "bf16")
    cache = fill_shared_cache(w, t, B, L, (L + 7) // 8 * 8, torch.bfloat16)
    row = torch.zeros((B, Hq, L), dtype=torch.float32, device="cuda")
    out = lb.lisa_attn_shared_decode(dev(t["prev"]), lb.Link(dev(t["qp"]), None, dev(w1), dev(w2), act=lb.ACT_RELU, integrate=integrate),
                                     cache, L=L, out_scores=row)
    O, R = oracle.decode_shared(f64(t["prev"]), f64(t["qp"])[:, 0], f64(t["kp"]), f64(t["v"]),
                                oracle.Link(None, None, f64(w1), f64(w2), r=w.r, act=ACT["relu"][1], integrate=integrate), np.full(B, L, np.int32))
    row_h = row.cpu().numpy().astype(np.float64)
    assert np.all(np.abs(R[:, :, at]) < 3e38) and np.abs(R[:, :, at]).max() > 1e36
    # sums of a few hundred products at 24 bits, whose terms are a few times larger than the result
    assert np.abs(row_h[:, :, at] - R[:, :, at]).max() <= 1e-5 * np.abs(R[:, :, at]).max()
    others = [j for j in range(L) if j not in at]
    assert_close(row_h[:, :, others], R[:, :, others], "f32", "row")
    assert_close(out[:, 0].float().cpu().numpy(), O, "bf16", "O")


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("Hq,Hkv,d,L", [(40, 40, 128, 600), (32, 8, 128, 257), (6, 3, 64, 130), (4, 4, 32, 7)])
def test_anchor_decode(dtype, Hq, Hkv, d, L):
    w = synth.Workload("adec", dtype, 2, L, Hq, Hkv, d, 8, 16, "relu", 1, True)
    tdt = torch.bfloat16 if dtype == "bf16" else torch.float32
    t = synth.decode_inputs(w, 6, B=2, L=L)
    L_cap = (L + 7) // 8 * 8
    cache = lb.KVCacheLayer(lb.CACHE_STANDARD, 2, Hkv, L_cap, d, dtype=tdt)
    lb.lisa_kvcache_append(cache, dev(t["k"]), dev(t["v"]))
    lens_h = np.array([L, (L + 1) // 2], dtype=np.int32)
    row = torch.full((2, Hq, L_cap), -7.0, dtype=torch.float32, device="cuda")
    out = lb.lisa_attn_anchor(dev(t["q0"]), cache=cache, L=L, seq_lens=torch.from_numpy(lens_h).cuda(), out_scores=row)
    O, R = oracle.decode_anchor(f64(t["q0"])[:, 0], f64(t["k"]), f64(t["v"]), lens_h)
    assert_close(out[:, 0].float().cpu().numpy(), O, dtype, "anchor decode O")
    row_h = row.cpu().numpy()
    for b in range(2):
        assert_close(row_h[b, :, :lens_h[b]], R[b, :, :lens_h[b]], "f32", "anchor score row")
        assert np.all(row_h[b, :, lens_h[b]:] == -7.0)


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_append_layouts_bit_exact(dtype):
    """Index work: the cache must hold exactly the appended values, K' transposed, at the right offsets."""
    B, Hkv, d, r, L_cap = 3, 2, 64, 21, 48
    g = torch.Generator().manual_seed(0)
    kp1, v1 = torch.randn(B, 20, Hkv, r, generator=g).to(dtype), torch.randn(B, 20, Hkv, d, generator=g).to(dtype)
    kp2, v2 = torch.randn(B, 1, Hkv, r, generator=g).to(dtype), torch.randn(B, 1, Hkv, d, generator=g).to(dtype)
    k1 = torch.randn(B, 20, Hkv, d, generator=g).to(dtype)
    sh = lb.KVCacheLayer(lb.CACHE_SHARED, B, Hkv, L_cap, d, r, dtype=dtype)
    st = lb.KVCacheLayer(lb.CACHE_STANDARD, B, Hkv, L_cap, d, dtype=dtype)
    lens = torch.tensor([20, 5, 0], dtype=torch.int32, device="cuda")
    lb.lisa_kvcache_append(sh, kp1.cuda(), v1.cuda())
    lb.lisa_kvcache_append(sh, kp2.cuda(), v2.cuda(), lens)
    lb.lisa_kvcache_append(st, k1.cuda(), v1.cuda())
    assert lb.lisa_check() == lb.OK
    exp_k = torch.zeros(B, Hkv, r, L_cap, dtype=dtype)
    exp_v = torch.zeros(B, Hkv, L_cap, d, dtype=dtype)
    exp_k[:, :, :, :20] = kp1.permute(0, 2, 3, 1)
    exp_v[:, :, :20] = v1.permute(0, 2, 1, 3)
    for b, off in enumerate([20, 5, 0]):
        exp_k[b, :, :, off] = kp2[b, 0]
        exp_v[b, :, off] = v2[b, 0]
    assert torch.equal(sh.k.cpu(), exp_k) and torch.equal(sh.v.cpu(), exp_v)
    assert torch.equal(st.k.cpu()[:, :, :20], k1.permute(0, 2, 1, 3)) and torch.equal(st.v.cpu()[:, :, :20], v1.permute(0, 2, 1, 3))


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("B,n,Hkv,r,d,before", [(2, 64, 3, 21, 128, 0), (1, 130, 2, 32, 64, 5), (3, 63, 5, 1, 32, 3), (2, 200, 1, 20, 128, 41)])
def test_append_prompt_layouts(dtype, B, n, Hkv, r, d, before):
    """Prompts around the 64-position tiles of the transposed copy, odd start positions, one run past the capacity."""
    g = torch.Generator().manual_seed(1)
    kp, v = torch.randn(B, n, Hkv, r, generator=g).to(dtype), torch.randn(B, n, Hkv, d, generator=g).to(dtype)
    L_cap = (before + n + 7) // 8 * 8
    sh = lb.KVCacheLayer(lb.CACHE_SHARED, B, Hkv, L_cap, d, r, dtype=dtype)
    lens = torch.tensor([before + (2 * b if b + 1 == B else 0) for b in range(B)], dtype=torch.int32)
    lb.lisa_kvcache_append(sh, kp.cuda(), v.cuda(), lens.cuda())
    exp_k, exp_v = torch.zeros(B, Hkv, r, L_cap, dtype=dtype), torch.zeros(B, Hkv, L_cap, d, dtype=dtype)
    for b, s in enumerate(lens.tolist()):
        m = min(n, L_cap - s)
        exp_k[b, :, :, s:s + m] = kp[b, :m].permute(1, 2, 0)
        exp_v[b, :, s:s + m] = v[b, :m].permute(1, 0, 2)
    assert torch.equal(sh.k.cpu(), exp_k) and torch.equal(sh.v.cpu(), exp_v)
    lb.lisa_check()   # (a run past the capacity was counted)


def test_append_beyond_capacity_is_dropped_and_reported():
    B, Hkv, d, r, L_cap = 1, 1, 32, 4, 8
    sh = lb.KVCacheLayer(lb.CACHE_SHARED, B, Hkv, L_cap, d, r)
    kp, v = torch.ones(B, 2, Hkv, r, dtype=torch.bfloat16, device="cuda"), torch.ones(B, 2, Hkv, d, dtype=torch.bfloat16, device="cuda")
    lb.lisa_kvcache_append(sh, kp, v, torch.tensor([7], dtype=torch.int32, device="cuda"))
    assert lb.lisa_check() == lb.ERR_INVALID_ARG      # one of two positions fell outside
    assert lb.lisa_check() == lb.OK                   # the report is consumed
    assert float(sh.v[0, 0, 7].float().sum()) == d and float(sh.k[0, 0, :, 7].float().sum()) == r


def test_decode_rejects_bad_arguments():
    w = D_SMALL
    t = synth.decode_inputs(w, 0, B=1, L=16)
    cache = fill_shared_cache(w, t, 1, 16, 16, torch.bfloat16)
    link = lb.Link(dev(t["qp"]), None, dev(t["w1"]), dev(t["w2"]))
    prev = dev(t["prev"])
    with pytest.raises(lb.LisaError) as e:
        lb.lisa_attn_shared_decode(prev, link, cache, L=17)
    assert e.value.status == lb.ERR_INVALID_ARG
    with pytest.raises(lb.LisaError) as e:
        lb.lisa_attn_shared_decode(prev, link, cache, L=16, out_scores=prev)
    assert e.value.status == lb.ERR_INVALID_ARG
    with pytest.raises(lb.LisaError) as e:
        lb.lisa_attn_shared_decode(prev, link, cache, L=16, workspace=torch.empty(16, dtype=torch.uint8, device="cuda"))
    assert e.value.status == lb.ERR_WORKSPACE


@pytest.mark.parametrize("Hq,Hkv,d,r,m,L", [(40, 40, 128, 21, 80, 700), (8, 2, 64, 21, 16, 300)])
def test_bf16_score_rows(Hq, Hkv, d, r, m, L):
    """Score rows handed between decode layers as bf16 (2 bytes per entry, the size Sec. 5.2 counts).  The layer reads the
    bf16 row exactly (the oracle gets the same rounded values), so its output stays within the usual bar; the row it writes
    is the oracle's row rounded to bf16 once more: relative 2^-8 at worst (half an ulp of 8 mantissa bits is 2^-9; the kernel's
    own fp32/tf32 arithmetic can move a value across a rounding boundary), which is what the hand-off costs per layer.
    The standard layer's row is checked the same way."""
    B = 2
    w = synth.Workload("rows16", "bf16", B, L, Hq, Hkv, d, r, m, "relu", 1, True)
    t = synth.decode_inputs(w, 8, B=B, L=L)
    L_cap = (L + 7) // 8 * 8
    lens_h = np.array([L, L // 2 + 1], dtype=np.int32)
    lens_d = torch.from_numpy(lens_h).cuda()
    prev16 = t["prev"].to(torch.bfloat16)
    cache = fill_shared_cache(w, t, B, L, L_cap, torch.bfloat16)
    link = lb.Link(dev(t["qp"]), None, dev(t["w1"]), dev(t["w2"]), act=lb.ACT_RELU)
    row = torch.full((B, Hq, L_cap), -7.0, dtype=torch.bfloat16, device="cuda")
    out = lb.lisa_attn_shared_decode(dev(prev16), link, cache, L=L, seq_lens=lens_d, out_scores=row)
    torch.cuda.synchronize()
    olink = oracle.Link(None, None, f64(t["w1"]), f64(t["w2"]), r=r, act=oracle.ACT_RELU)
    O, R = oracle.decode_shared(f64(prev16), f64(t["qp"])[:, 0], f64(t["kp"]), f64(t["v"]), olink, lens_h)
    assert_close(out[:, 0].float().cpu().numpy(), O, "bf16", "decode O from a bf16 row")
    row_h = row.float().cpu().numpy()
    for b in range(B):
        got, ref = row_h[b, :, :lens_h[b]], R[b, :, :lens_h[b]]
        assert np.all(np.abs(got - ref) <= 2.0 ** -8 * np.abs(ref) + 3e-3), "bf16 row beyond one rounding of the oracle's row"
        assert np.all(row_h[b, :, lens_h[b]:] == -7.0), "row written beyond the sequence length"
    # standard layer emitting a bf16 row
    st = lb.KVCacheLayer(lb.CACHE_STANDARD, B, Hkv, L_cap, d)
    lb.lisa_kvcache_append(st, dev(t["k"]), dev(t["v"]))
    row0 = torch.full((B, Hq, L_cap), -7.0, dtype=torch.bfloat16, device="cuda")
    out0 = lb.lisa_attn_anchor(dev(t["q0"]), cache=st, L=L, seq_lens=lens_d, out_scores=row0)
    O0, R0 = oracle.decode_anchor(f64(t["q0"])[:, 0], f64(t["k"]), f64(t["v"]), lens_h)
    assert_close(out0[:, 0].float().cpu().numpy(), O0, "bf16", "standard decode O with a bf16 row")
    r0 = row0.float().cpu().numpy()
    for b in range(B):
        got, ref = r0[b, :, :lens_h[b]], R0[b, :, :lens_h[b]]
        assert np.all(np.abs(got - ref) <= 2.0 ** -8 * np.abs(ref) + 1e-4)
        assert np.all(r0[b, :, lens_h[b]:] == -7.0)
    assert lb.lisa_check() == lb.OK


def test_multi_layer_cache_handle_matches_per_layer_caches():
    """lisa_kvcache_init carves one buffer into per-layer caches; lisa_kvcache_append_layer on it and a decode step on one of its
    layers give bit for bit what separately allocated per-layer caches give."""
    B, L, Hq, Hkv, d, r, m = 2, 200, 8, 2, 64, 21, 16
    w = synth.Workload("handle", "bf16", B, L, Hq, Hkv, d, r, m, "relu", 1, True)
    t = synth.decode_inputs(w, 12, B=B, L=L)
    L_cap = 208
    whole = lb.KVCache([lb.CACHE_STANDARD, lb.CACHE_SHARED, lb.CACHE_SHARED], B, Hkv, L_cap, d, r)
    whole.append(0, dev(t["k"]), dev(t["v"]))
    whole.append(1, dev(t["kp"]), dev(t["v"]))
    first = 152                                                  # layer 2 in two pieces, the second at an offset (its rows start 16-byte aligned)
    whole.append(2, dev(t["kp"])[:, :first], dev(t["v"])[:, :first])
    before = torch.full((B,), first, dtype=torch.int32, device="cuda")
    whole.append(2, dev(t["kp"])[:, first:], dev(t["v"])[:, first:], before)
    std = lb.KVCacheLayer(lb.CACHE_STANDARD, B, Hkv, L_cap, d)
    sh = lb.KVCacheLayer(lb.CACHE_SHARED, B, Hkv, L_cap, d, r)
    lb.lisa_kvcache_append(std, dev(t["k"]), dev(t["v"]))
    lb.lisa_kvcache_append(sh, dev(t["kp"]), dev(t["v"]))
    torch.cuda.synchronize()
    assert torch.equal(whole.layer(0).k, std.k) and torch.equal(whole.layer(0).v, std.v)
    for l in (1, 2):
        assert torch.equal(whole.layer(l).k, sh.k) and torch.equal(whole.layer(l).v, sh.v)
    link = lb.Link(dev(t["qp"]), None, dev(t["w1"]), dev(t["w2"]), act=lb.ACT_RELU)
    a = lb.lisa_attn_shared_decode(dev(t["prev"]), link, whole.layer(2), L=L)
    b = lb.lisa_attn_shared_decode(dev(t["prev"]), link, sh, L=L)
    assert torch.equal(a, b)
    with pytest.raises(lb.LisaError):
        whole.append(3, dev(t["kp"]), dev(t["v"]))               # no such layer
    assert lb.lisa_check() == lb.OK


@pytest.mark.parametrize("Hq,Hkv,m,integrate,B,L", [(32, 8, 64, lb.INTEGRATE_ADD, 66, 600), (40, 40, 80, lb.INTEGRATE_ADD, 34, 1150),
                                                     (32, 32, 128, lb.INTEGRATE_CONCAT, 34, 1100), (32, 8, 72, lb.INTEGRATE_ADD, 34, 1100)])
def test_ragged_batches_whose_chunks_are_dealt(Hq, Hkv, m, integrate, B, L):
    """Grids of 297..444 CTAs (on 148 SMs) of a ragged batch: the chunks that hold positions are numbered on the device.  Lengths on and around
    the chunk's edges, sequences past the first 32 and 64; the aligners on tf32 and on bf16 terms; then the standard layer of the same lengths."""
    lens = np.random.default_rng(B).integers(1, L + 1, B).astype(np.int32)
    lens[[0, 1, 2, 3, 31, 32, 33, B - 1]] = [1, 127, 128, 129, L, 256, 1, L - 1]
    w = synth.Workload("dealt", "bf16", B, L, Hq, Hkv, 128, 21, m, "relu", 1, True)
    run_shared_decode(w, B, L, lens=lens, seed=3, integrate=integrate)
    if Hkv == 8:
        t = synth.decode_inputs(w, 3, B=B, L=L)
        cache = lb.KVCacheLayer(lb.CACHE_STANDARD, B, Hkv, (L + 7) // 8 * 8, 128)
        lb.lisa_kvcache_append(cache, dev(t["k"]), dev(t["v"]))
        row = torch.full((B, Hq, (L + 7) // 8 * 8), -7.0, dtype=torch.float32, device="cuda")
        out = lb.lisa_attn_anchor(dev(t["q0"]), cache=cache, L=L, seq_lens=torch.from_numpy(lens).cuda(), out_scores=row)
        O, R = oracle.decode_anchor(f64(t["q0"])[:, 0], f64(t["k"]), f64(t["v"]), lens)
        assert_close(out[:, 0].float().cpu().numpy(), O, "bf16", "standard O")
        for b in range(B):
            assert_close(row.cpu().numpy()[b, :, :lens[b]], R[b, :, :lens[b]], "bf16", "standard row")


@pytest.mark.parametrize("Hq,Hkv,d,m,B,L", [
    (32, 8, 128, 64, 4, 256), (32, 8, 128, 64, 4, 257),        # 1024 positions and more
    (32, 32, 128, 64, 6, 60), (32, 32, 128, 64, 7, 60),        # 192 and 224 merges on 148 SMs: one and a half times as many lie between
    (40, 40, 128, 80, 5, 128), (40, 40, 128, 80, 6, 128),
    (8, 2, 64, 16, 3, 300), (8, 2, 64, 16, 4, 300)])           # the general chunk kernels
def test_layers_enqueued_behind_one_another_equal_layers_one_by_one(Hq, Hkv, d, m, B, L):
    """Where the merge lets the kernels behind it in at its start and where behind its wait: append, standard layer, append, shared layers with one
    workspace and no wait between them give the bytes of the same calls with the GPU waited for after each, and the last layer is the oracle's."""
    w = synth.Workload("behind", "bf16", B, L, Hq, Hkv, d, 21, m, "relu", 1, True)
    t = synth.decode_inputs(w, 5, B=B, L=L)
    L_cap = (L + 15) // 8 * 8
    ws = torch.empty(lb.decode_workspace_bytes(B, Hq, d, L), dtype=torch.uint8, device="cuda")
    before = torch.full((B,), L - 1, dtype=torch.int32, device="cuda")
    x = {k: dev(v) for k, v in t.items()}

    def step(wait):
        def done(y=None):
            if wait:
                torch.cuda.synchronize()
            return y
        st = lb.KVCacheLayer(lb.CACHE_STANDARD, B, Hkv, L_cap, d)
        sh = [lb.KVCacheLayer(lb.CACHE_SHARED, B, Hkv, L_cap, d, w.r) for _ in range(2)]
        rows = [torch.zeros((B, Hq, L_cap), dtype=torch.float32, device="cuda") for _ in range(2)]
        for cache, k in [(st, "k")] + [(c, "kp") for c in sh]:
            lb.lisa_kvcache_append(cache, x[k][:, :L - 1].contiguous(), x["v"][:, :L - 1].contiguous())
        new = {k: x[k][:, L - 1:].contiguous() for k in ("k", "kp", "v")}
        torch.cuda.synchronize()
        outs = []
        done(lb.lisa_kvcache_append(st, new["k"], new["v"], before))
        outs.append(done(lb.lisa_attn_anchor(x["q0"], cache=st, L=L, out_scores=rows[0], workspace=ws)))
        for i in range(2):
            done(lb.lisa_kvcache_append(sh[i], new["kp"], new["v"], before))
            link = lb.Link(x["qp"], None, x["w1"], x["w2"], act=lb.ACT_RELU)
            outs.append(done(lb.lisa_attn_shared_decode(rows[i], link, sh[i], L=L, out_scores=rows[1] if i == 0 else None, workspace=ws)))
        torch.cuda.synchronize()
        return outs + rows

    ref = step(True)
    for _ in range(3):
        assert all(torch.equal(a, b) for a, b in zip(step(False), ref))
    lens = np.full((B,), L, dtype=np.int32)
    O0, R0 = oracle.decode_anchor(f64(t["q0"])[:, 0], f64(t["k"]), f64(t["v"]), lens)
    assert_close(ref[0][:, 0].float().cpu().numpy(), O0, "bf16", "standard O")
    olink = oracle.Link(None, None, f64(t["w1"]), f64(t["w2"]), r=w.r, act=oracle.ACT_RELU)
    for i in range(2):
        O, R = oracle.decode_shared(R0 if i == 0 else ref[4][:, :, :L].cpu().numpy().astype(np.float64), f64(t["qp"])[:, 0], f64(t["kp"]), f64(t["v"]), olink, lens)
        assert_close(ref[1 + i][:, 0].float().cpu().numpy(), O, "bf16", "shared O %d" % i)
    assert lb.lisa_check() == lb.OK
