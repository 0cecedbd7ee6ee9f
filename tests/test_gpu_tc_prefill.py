"""GPU parity of the tensor-core prefill kernels (head width 128, bf16) against the CPU oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2408_01890_b200 import binding as lb
from paper_2408_01890_b200 import synth
from helpers import assert_close, dev, f64, make_links

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,N,Hq,Hkv", [(1, 128, 2, 2), (1, 256, 4, 2), (2, 300, 4, 1), (1, 1, 2, 2), (1, 1000, 8, 8)])
def test_anchor_prefill_tensor_core(B, N, Hq, Hkv):
    w = synth.Workload("tc_anchor", "bf16", B, N, Hq, Hkv, 128, 21, 64, "relu", 0)
    t = synth.prefill_inputs(w, 1)
    n0 = lb.lisa_kernel_launches()
    got = lb.lisa_attn_anchor(dev(t["q0"]), dev(t["k0"]), dev(t["v0"]))
    torch.cuda.synchronize()
    assert lb.lisa_kernel_launches() - n0 == 1
    assert lb.lisa_check() == lb.OK
    ref = oracle.prefill_full(f64(t["q0"]), f64(t["k0"]), f64(t["v0"]), [])
    assert_close(got.float().cpu().numpy(), ref, "bf16", "tensor-core anchor prefill")
    lb.lisa_force_general_kernels(True)
    try:
        gen = lb.lisa_attn_anchor(dev(t["q0"]), dev(t["k0"]), dev(t["v0"]))
    finally:
        lb.lisa_force_general_kernels(False)
    assert_close(gen.float().cpu().numpy(), ref, "bf16", "general anchor prefill")


def run_tc_shared(B, N, Hkv, chain, act, seed=0, bias=False, r=21):
    w = synth.Workload("tc_shared", "bf16", B, N, 32, Hkv, 128, r, 64, act, chain)
    t = synth.prefill_inputs(w, seed)
    if bias:
        for k in range(1, chain + 1):
            t[f"b1_{k}"] = synth.as_dtype(synth.normal(f"b1_{k}", (64,), seed, std=0.5), "bf16")
            t[f"b2_{k}"] = synth.as_dtype(synth.normal(f"b2_{k}", (32,), seed, std=0.5), "bf16")
    dl, ol = make_links(t, chain, act, bias=bias)
    n0 = lb.lisa_kernel_launches()
    got = lb.lisa_attn_shared_prefill(dev(t["q0"]), dev(t["k0"]), dl, dev(t[f"v{chain}"]))
    torch.cuda.synchronize()
    if chain <= 3:
        assert lb.lisa_kernel_launches() - n0 == chain + 3  # pack, one emit per plane, align, attention
    assert lb.lisa_check() == lb.OK
    ref = oracle.prefill_full(f64(t["q0"]), f64(t["k0"]), f64(t[f"v{chain}"]), ol)
    return assert_close(got.float().cpu().numpy(), ref, "bf16", "tensor-core shared prefill N=%d c=%d" % (N, chain))


@pytest.mark.parametrize("B,N,Hkv,chain,act", [(1, 128, 32, 1, "relu"), (1, 256, 32, 1, "silu"), (2, 300, 8, 1, "relu"),
                                                 (1, 200, 32, 2, "relu"), (1, 513, 8, 3, "silu"), (1, 130, 32, 4, "none"), (1, 260, 32, 3, "none")])
def test_shared_prefill_tensor_core(B, N, Hkv, chain, act):
    run_tc_shared(B, N, Hkv, chain, act)


@pytest.mark.parametrize("B,N,Hkv,chain,act,hq", [(1, 300, 8, 3, "relu", 32), (2, 200, 32, 2, "silu", 32), (1, 130, 32, 1, "relu", 32),
                                                    (1, 150, 4, 3, "relu", 8)])
def test_shared_prefill_chain(B, N, Hkv, chain, act, hq):
    """All layers of a chain in one pass: layer k's output equals the oracle's layer at depth k+1 with its own V.
    Hq = 32 runs the tensor-core kernels (every link's output stored by one aligner pass), Hq = 8 the layer-by-layer route."""
    w = synth.Workload("tc_chain", "bf16", B, N, hq, Hkv, 128, 21, 2 * hq, act, chain)
    t = synth.prefill_inputs(w, 7)
    dl, ol = make_links(t, chain, act)
    vs = [dev(t[f"v{k}"]) for k in range(1, chain + 1)]
    n0 = lb.lisa_kernel_launches()
    outs = lb.lisa_attn_shared_prefill_chain(dev(t["q0"]), dev(t["k0"]), dl, vs)
    torch.cuda.synchronize()
    if hq == 32:   # one pack + emits (chain) + one aligner + one attention per layer
        assert lb.lisa_kernel_launches() - n0 == 1 + chain + 1 + chain
    assert lb.lisa_check() == lb.OK
    for k in range(chain):
        ref = oracle.prefill_full(f64(t["q0"]), f64(t["k0"]), f64(t[f"v{k + 1}"]), ol[:k + 1])
        assert_close(outs[k].float().cpu().numpy(), ref, "bf16", "chain prefill N=%d layer %d of %d" % (N, k + 1, chain))


def test_shared_prefill_chain_rejects_bad_arguments():
    w = synth.Workload("tc_chain", "bf16", 1, 130, 32, 32, 128, 21, 64, "relu", 2)
    t = synth.prefill_inputs(w, 1)
    dl, _ = make_links(t, 2, "relu")
    vs = [dev(t["v1"]), dev(t["v2"])]
    with pytest.raises(lb.LisaError):      # workspace too small
        lb.lisa_attn_shared_prefill_chain(dev(t["q0"]), dev(t["k0"]), dl, vs, workspace=torch.empty(1024, dtype=torch.uint8, device="cuda"))
    with pytest.raises(lb.LisaError):      # 32 query heads do not divide over 3 key heads
        lb.lisa_attn_shared_prefill_chain(dev(t["q0"]), dev(t["k0"])[:, :, :3], dl, vs)
    assert lb.lisa_check() == lb.OK


def test_shared_prefill_tensor_core_bias_and_rank():
    run_tc_shared(1, 260, 32, 2, "relu", seed=3, bias=True, r=32)
    run_tc_shared(1, 140, 32, 1, "silu", seed=4, bias=True, r=8)


def test_bounded_wait_runs_out_and_the_context_survives():
    """A device-side wait that nothing satisfies gives up by itself: the status word reports it once (LISA_ERR_TIMEOUT),
    the next check is clean, and a tensor-core prefill launched right after still matches the oracle."""
    assert lb.lisa_check() == lb.OK
    lb.lisa_debug_wait_timeout(1000000)          # about half a millisecond of waiting, then the kernel returns
    assert lb.lisa_check() == lb.ERR_TIMEOUT
    assert lb.lisa_check() == lb.OK
    run_tc_shared(1, 256, 32, 1, "relu", seed=5)
    with pytest.raises(lb.LisaError):
        lb.lisa_debug_wait_timeout(10 ** 12)     # limits beyond 1e8 cycles are refused before anything is launched


@pytest.mark.parametrize("integrate,layers,chain,r,bias", [
    (lb.INTEGRATE_ADD, 1, 1, 32, True),       # one linear 32 x 32 layer over the heads, r = 32
    (lb.INTEGRATE_ADD, 1, 3, 21, False),
    (lb.INTEGRATE_PLUS, 2, 1, 20, False),     # no FFN: A_n = A_{n-1} + A_Delta (Sec. 6.3's variant for pre-trained sharing)
    (lb.INTEGRATE_PLUS, 2, 3, 21, False)])
def test_variants_without_a_hidden_layer_run_on_the_tensor_cores(integrate, layers, chain, r, bias):
    """32 heads, d = 128: the one-layer aligner and the FFN-free variant take the tensor-core path (seen in the launch count:
    pack, one emit per plane, align, attention) and match the oracle like the two-layer FFN does."""
    B, N, Hkv = 1, 300, 8
    w = synth.Workload("tc_variant", "bf16", B, N, 32, Hkv, 128, r, 32, "none", chain)
    t = synth.prefill_inputs(w, 13)
    for k in range(1, chain + 1):
        t[f"w1_{k}"] = synth.as_dtype(synth.normal(f"w1_{k}", (32, 32), 13, std=32 ** -0.5), "bf16")
        t[f"b1_{k}"] = synth.as_dtype(synth.normal(f"b1_{k}", (32,), 13, std=0.5), "bf16")
    dl, ol = make_links(t, chain, "none", integrate, layers, bias)
    n0 = lb.lisa_kernel_launches()
    got = lb.lisa_attn_shared_prefill(dev(t["q0"]), dev(t["k0"]), dl, dev(t[f"v{chain}"]))
    torch.cuda.synchronize()
    assert lb.lisa_kernel_launches() - n0 == chain + 3
    assert lb.lisa_check() == lb.OK
    ref = oracle.prefill_full(f64(t["q0"]), f64(t["k0"]), f64(t[f"v{chain}"]), ol)
    assert_close(got.float().cpu().numpy(), ref, "bf16", "tensor-core prefill, variant without a hidden layer")


def concat_inputs(B, N, Hkv, chain, m, act, layers, r, seed, bias):
    w = synth.Workload("tc_concat", "bf16", B, N, 32, Hkv, 128, r, m, act, chain)
    t = synth.prefill_inputs(w, seed)
    mm = 32 if layers == 1 else m
    for k in range(1, chain + 1):
        t[f"w1_{k}"] = synth.as_dtype(synth.normal(f"w1_{k}", (64, mm), seed, std=64 ** -0.5), "bf16")
        t[f"w2_{k}"] = synth.as_dtype(synth.normal(f"w2_{k}", (mm, 32), seed, std=mm ** -0.5), "bf16")
        t[f"b1_{k}"] = synth.as_dtype(synth.normal(f"b1_{k}", (mm,), seed, std=0.5), "bf16")
        t[f"b2_{k}"] = synth.as_dtype(synth.normal(f"b2_{k}", (32,), seed, std=0.5), "bf16")
    return t


@pytest.mark.parametrize("B,N,Hkv,chain,m,act,layers,r,bias", [
    (1, 300, 32, 1, 256, "relu", 2, 20, False),    # the paper's complete model: FFN 64 x 256, 256 x 32, ReLU, r = 20
    (2, 200, 8, 2, 64, "silu", 2, 21, True),
    (1, 260, 32, 3, 200, "relu", 2, 21, True),     # hidden width that is not a multiple of 64
    (1, 300, 8, 1, 32, "none", 1, 32, True),       # one linear 64 x 32 layer, r = 32
    (1, 150, 32, 2, 32, "none", 1, 21, False)])
def test_concatenating_integrate_runs_on_the_tensor_cores(B, N, Hkv, chain, m, act, layers, r, bias):
    """Integrate by concatenation (Sec. 5.1, the overview's complete model): [A_{n-1}; A_Delta] through the FFN, 32 heads,
    d = 128, on the tensor-core path (launches: pack, A_0 and one difference plane per link, one aligner pass per link,
    attention) against the oracle."""
    t = concat_inputs(B, N, Hkv, chain, m, act, layers, r, 17, bias)
    dl, ol = make_links(t, chain, act, lb.INTEGRATE_CONCAT, layers, bias)
    n0 = lb.lisa_kernel_launches()
    got = lb.lisa_attn_shared_prefill(dev(t["q0"]), dev(t["k0"]), dl, dev(t[f"v{chain}"]))
    torch.cuda.synchronize()
    assert lb.lisa_kernel_launches() - n0 == 2 * chain + 3
    assert lb.lisa_check() == lb.OK
    ref = oracle.prefill_full(f64(t["q0"]), f64(t["k0"]), f64(t[f"v{chain}"]), ol)
    assert_close(got.float().cpu().numpy(), ref, "bf16", "tensor-core prefill, concatenating integrate")


def test_concatenating_chain_in_one_pass():
    """lisa_attn_shared_prefill_chain with the concatenating Integrate: every layer of the chain against the oracle."""
    B, N, Hkv, chain = 1, 300, 8, 3
    t = concat_inputs(B, N, Hkv, chain, 256, "relu", 2, 20, 19, False)
    dl, ol = make_links(t, chain, "relu", lb.INTEGRATE_CONCAT, 2, False)
    n0 = lb.lisa_kernel_launches()
    outs = lb.lisa_attn_shared_prefill_chain(dev(t["q0"]), dev(t["k0"]), dl, [dev(t[f"v{k}"]) for k in range(1, chain + 1)])
    torch.cuda.synchronize()
    assert lb.lisa_kernel_launches() - n0 == 1 + (1 + chain) + chain + chain   # pack, planes, aligner passes, one attention per layer
    for k in range(chain):
        ref = oracle.prefill_full(f64(t["q0"]), f64(t["k0"]), f64(t[f"v{k + 1}"]), ol[:k + 1])
        assert_close(outs[k].float().cpu().numpy(), ref, "bf16", "concatenating chain, layer %d" % (k + 1))
    assert lb.lisa_check() == lb.OK


def link_inputs(B, N, Hq, Hkv, chain, m, act, layers, r, seed, bias):
    w = synth.Workload("tc_link", "bf16", B, N, Hq, Hkv, 128, r, m, act, chain)
    t = synth.prefill_inputs(w, seed)
    mm = Hq if layers == 1 else m
    for k in range(1, chain + 1):
        t[f"w1_{k}"] = synth.as_dtype(synth.normal(f"w1_{k}", (Hq, mm), seed, std=Hq ** -0.5), "bf16")
        t[f"w2_{k}"] = synth.as_dtype(synth.normal(f"w2_{k}", (mm, Hq), seed, std=mm ** -0.5), "bf16")
        t[f"b1_{k}"] = synth.as_dtype(synth.normal(f"b1_{k}", (mm,), seed, std=0.5), "bf16")
        t[f"b2_{k}"] = synth.as_dtype(synth.normal(f"b2_{k}", (Hq,), seed, std=0.5), "bf16")
    return t


@pytest.mark.parametrize("B,N,Hq,Hkv,chain,m,act,integrate,layers,r,bias", [
    (1, 300, 40, 40, 1, 80, "relu", lb.INTEGRATE_ADD, 2, 21, False),    # the LLaMA2-13B layer: 40 heads, FFN 40 -> 80 -> 40
    (2, 200, 40, 8, 2, 80, "silu", lb.INTEGRATE_ADD, 2, 20, True),
    (1, 260, 40, 40, 3, 200, "relu", lb.INTEGRATE_ADD, 2, 21, True),     # hidden width over several chunks, not a multiple of 64
    (1, 150, 40, 40, 2, 48, "relu", lb.INTEGRATE_ADD, 2, 32, True),      # hidden width within one 64-unit chunk
    (1, 300, 40, 8, 2, 40, "none", lb.INTEGRATE_ADD, 1, 21, True),       # one linear 40 x 40 layer
    (1, 200, 40, 40, 3, 40, "none", lb.INTEGRATE_PLUS, 2, 21, False),    # no FFN
    (1, 300, 32, 8, 2, 128, "relu", lb.INTEGRATE_ADD, 2, 21, True),      # 32 heads with a hidden layer wider than 64
    (1, 513, 32, 32, 1, 256, "silu", lb.INTEGRATE_ADD, 2, 21, False)])
def test_link_by_link_aligner_runs_on_the_tensor_cores(B, N, Hq, Hkv, chain, m, act, integrate, layers, r, bias):
    """Adding links at 40 heads, or at 32 heads with a hidden layer wider than 64: one aligner launch per link on the
    tensor-core path (launches: pack, A_0 and one difference plane per link below the top, one aligner pass per link,
    attention) against the oracle."""
    t = link_inputs(B, N, Hq, Hkv, chain, m, act, layers, r, 23, bias)
    dl, ol = make_links(t, chain, act, integrate, layers, bias)
    n0 = lb.lisa_kernel_launches()
    got = lb.lisa_attn_shared_prefill(dev(t["q0"]), dev(t["k0"]), dl, dev(t[f"v{chain}"]))
    torch.cuda.synchronize()
    assert lb.lisa_kernel_launches() - n0 == 2 * chain + 2
    assert lb.lisa_check() == lb.OK
    ref = oracle.prefill_full(f64(t["q0"]), f64(t["k0"]), f64(t[f"v{chain}"]), ol)
    assert_close(got.float().cpu().numpy(), ref, "bf16", "tensor-core prefill, link-by-link aligner, %d heads" % Hq)


def test_link_by_link_chain_in_one_pass():
    """lisa_attn_shared_prefill_chain at the LLaMA2-13B layer shape (40 heads, 40 -> 80 -> 40): every layer of the chain."""
    B, N, Hq, Hkv, chain = 1, 300, 40, 40, 3
    t = link_inputs(B, N, Hq, Hkv, chain, 80, "relu", 2, 21, 29, True)
    dl, ol = make_links(t, chain, "relu", lb.INTEGRATE_ADD, 2, True)
    n0 = lb.lisa_kernel_launches()
    outs = lb.lisa_attn_shared_prefill_chain(dev(t["q0"]), dev(t["k0"]), dl, [dev(t[f"v{k}"]) for k in range(1, chain + 1)])
    torch.cuda.synchronize()
    assert lb.lisa_kernel_launches() - n0 == 1 + chain + chain + chain   # pack, planes, aligner passes, one attention per layer
    for k in range(chain):
        ref = oracle.prefill_full(f64(t["q0"]), f64(t["k0"]), f64(t[f"v{k + 1}"]), ol[:k + 1])
        assert_close(outs[k].float().cpu().numpy(), ref, "bf16", "link-by-link chain at 40 heads, layer %d" % (k + 1))
    assert lb.lisa_check() == lb.OK


@pytest.mark.parametrize("B,N,Hq,Hkv,chain,m,act,integrate,layers,bias", [
    (2, 300, 32, 8, 3, 64, "relu", lb.INTEGRATE_ADD, 2, False),     # the cfg3 layer shape
    (1, 513, 32, 32, 6, 64, "silu", lb.INTEGRATE_ADD, 2, True),     # a run of six shared layers: deeper than the recomputing kernels take
    (1, 200, 40, 40, 3, 80, "relu", lb.INTEGRATE_ADD, 2, True),     # LLaMA2-13B layer shape (link-by-link aligner)
    (1, 260, 32, 8, 2, 32, "none", lb.INTEGRATE_ADD, 1, True),      # one linear layer
    (1, 130, 32, 32, 3, 64, "none", lb.INTEGRATE_PLUS, 2, False)])  # no FFN
def test_carried_scores_layer_by_layer(B, N, Hq, Hkv, chain, m, act, integrate, layers, bias):
    """lisa_attn_shared_prefill_carry: every layer of a chain takes A_{n-1} from the scores buffer the layer before left
    (Sec. 5.1) and must equal the oracle's layer at that depth; only the first layer computes the anchor's scores (seen in
    the launch counts: pack, emit, align, attention for the first layer; pack, align, attention afterwards)."""
    t = link_inputs(B, N, Hq, Hkv, chain, m, act, layers, 21, 31, bias)
    dl, ol = make_links(t, chain, act, integrate, layers, bias)
    scores = torch.full((lb.lisa_prefill_scores_bytes(B, N, Hq),), 0xFF, dtype=torch.uint8, device="cuda")   # NaN patterns where nothing was written
    q0, k0 = dev(t["q0"]), dev(t["k0"])
    for k in range(chain):
        v = dev(t[f"v{k + 1}"])
        n0 = lb.lisa_kernel_launches()
        if k == 0:
            got = lb.lisa_attn_shared_prefill_carry(q0, k0, dl[0], v, scores, first=True, keep=chain > 1)
        else:
            got = lb.lisa_attn_shared_prefill_carry(None, None, dl[k], v, scores, first=False, keep=k + 1 < chain, out=torch.empty_like(q0))
        torch.cuda.synchronize()
        assert lb.lisa_kernel_launches() - n0 == (4 if k == 0 else 3)
        assert lb.lisa_check() == lb.OK
        ref = oracle.prefill_full(f64(t["q0"]), f64(t["k0"]), f64(t[f"v{k + 1}"]), ol[:k + 1])
        assert_close(got.float().cpu().numpy(), ref, "bf16", "carried scores, layer %d of %d, %d heads" % (k + 1, chain, Hq))


def test_carried_scores_rejects_bad_arguments():
    B, N, Hq, Hkv = 1, 130, 32, 32
    t = link_inputs(B, N, Hq, Hkv, 1, 64, "relu", 2, 21, 33, False)
    dl, _ = make_links(t, 1, "relu")
    q0, k0, v = dev(t["q0"]), dev(t["k0"]), dev(t["v1"])
    need = lb.lisa_prefill_scores_bytes(B, N, Hq)
    assert need == B * Hq * 256 * 256 * 2
    small = torch.empty(need - 1, dtype=torch.uint8, device="cuda")
    with pytest.raises(lb.LisaError) as ei:
        lb.lisa_attn_shared_prefill_carry(q0, k0, dl[0], v, small, first=True, keep=True)
    assert ei.value.status == lb.ERR_INVALID_ARG
    scores = torch.empty(need, dtype=torch.uint8, device="cuda")
    wide = link_inputs(B, N, Hq, Hkv, 1, 320, "relu", 2, 21, 33, False)
    dw, _ = make_links(wide, 1, "relu")
    with pytest.raises(lb.LisaError) as ei:   # hidden width beyond the tensor-core aligners: no carried form
        lb.lisa_attn_shared_prefill_carry(q0, k0, dw[0], v, scores, first=True, keep=True)
    assert ei.value.status == lb.ERR_UNSUPPORTED
    assert lb.lisa_check() == lb.OK


def test_carried_scores_from_host_memory():
    """lisa_attn_shared_prefill_carry_host: the layer's tensors come from host memory and its output goes back there; the scores
    stay on the device from layer to layer.  Same results as the device-memory calls."""
    B, N, Hq, Hkv, chain = 1, 300, 32, 8, 3
    t = link_inputs(B, N, Hq, Hkv, chain, 64, "relu", 2, 21, 37, True)
    dl, ol = make_links(t, chain, "relu", lb.INTEGRATE_ADD, 2, True)
    scores = torch.empty(lb.lisa_prefill_scores_bytes(B, N, Hq), dtype=torch.uint8, device="cuda")
    scores2 = torch.empty_like(scores)
    for k in range(chain):
        hl = lb.Link(t[f"qp{k + 1}"], t[f"kp{k + 1}"], t[f"w1_{k + 1}"], t[f"w2_{k + 1}"], t[f"b1_{k + 1}"], t[f"b2_{k + 1}"], act=lb.ACT_RELU)
        out_h = torch.empty_like(t["q0"])
        need = lb.lisa_carry_host_arena_bytes(t["q0"], t["k0"], hl, t[f"v{k + 1}"], out_h, scores2, first=k == 0)
        arena = torch.empty(need, dtype=torch.uint8, device="cuda")
        lb.lisa_attn_shared_prefill_carry_host(t["q0"], t["k0"], hl, t[f"v{k + 1}"], out_h, scores2, arena, first=k == 0, keep=k + 1 < chain)
        got = lb.lisa_attn_shared_prefill_carry(dev(t["q0"]), dev(t["k0"]), dl[k], dev(t[f"v{k + 1}"]), scores, first=k == 0, keep=k + 1 < chain)
        torch.cuda.synchronize()
        assert torch.equal(out_h, got.cpu())
        ref = oracle.prefill_full(f64(t["q0"]), f64(t["k0"]), f64(t[f"v{k + 1}"]), ol[:k + 1])
        assert_close(out_h.float().numpy(), ref, "bf16", "carried scores from host memory, layer %d" % (k + 1))
        if k > 0:   # past the first layer the arena holds no copy of q0, k0
            assert need < lb.lisa_carry_host_arena_bytes(t["q0"], t["k0"], hl, t[f"v{k + 1}"], out_h, scores2, first=True)
    assert lb.lisa_check() == lb.OK


@pytest.mark.parametrize("B,N,Hkv,chain,m,act,layers,r,bias", [
    (1, 300, 32, 3, 256, "relu", 2, 20, False),    # a run of three of the paper's complete layers (64 x 256, 256 x 32, ReLU, r = 20)
    (2, 200, 8, 4, 64, "silu", 2, 21, True),
    (1, 260, 8, 2, 32, "none", 1, 32, True)])      # one linear 64 x 32 layer
def test_carried_scores_concatenating_integrate(B, N, Hkv, chain, m, act, layers, r, bias):
    """The concatenating Integrate with carried scores: the aligner reads A_{n-1} from the scores buffer and the layer's
    difference from a plane of the wave, leaves A_n in the buffer, and hands the attention kernel its copy through the
    difference's plane (launches: pack, [A_0,] the difference, align, attention)."""
    t = concat_inputs(B, N, Hkv, chain, m, act, layers, r, 41, bias)
    dl, ol = make_links(t, chain, act, lb.INTEGRATE_CONCAT, layers, bias)
    scores = torch.full((lb.lisa_prefill_scores_bytes(B, N, 32),), 0xFF, dtype=torch.uint8, device="cuda")
    q0, k0 = dev(t["q0"]), dev(t["k0"])
    for k in range(chain):
        n0 = lb.lisa_kernel_launches()
        got = lb.lisa_attn_shared_prefill_carry(q0 if k == 0 else None, k0 if k == 0 else None, dl[k], dev(t[f"v{k + 1}"]), scores,
                                                first=k == 0, keep=k + 1 < chain, out=torch.empty_like(q0))
        torch.cuda.synchronize()
        assert lb.lisa_kernel_launches() - n0 == (5 if k == 0 else 4)
        assert lb.lisa_check() == lb.OK
        ref = oracle.prefill_full(f64(t["q0"]), f64(t["k0"]), f64(t[f"v{k + 1}"]), ol[:k + 1])
        assert_close(got.float().cpu().numpy(), ref, "bf16", "carried scores, concatenating integrate, layer %d of %d" % (k + 1, chain))


def test_carried_scores_concatenating_integrate_in_two_waves():
    """B = 4, N = 1600: the plane of the difference exceeds one wave's budget, so the eleven first query tiles and the two last ones go out as two waves
    on two streams, each with a plane of its own, over one scores buffer.  Launches: pack, and per wave [A_0,] the difference, align, attention."""
    B, N, chain = 4, 1600, 2
    t = concat_inputs(B, N, 8, chain, 64, "relu", 2, 20, 19, True)
    dl, ol = make_links(t, chain, "relu", lb.INTEGRATE_CONCAT, 2, True)
    scores = torch.full((lb.lisa_prefill_scores_bytes(B, N, 32),), 0xFF, dtype=torch.uint8, device="cuda")
    q0, k0 = dev(t["q0"]), dev(t["k0"])
    ri = np.concatenate([np.arange(0, 1408, 97), np.arange(1407, 1411), np.arange(1535, 1538), np.arange(N - 3, N)]).astype(np.int32)
    rb = np.full(ri.shape, B - 1, dtype=np.int32)
    for k in range(chain):
        n0 = lb.lisa_kernel_launches()
        got = lb.lisa_attn_shared_prefill_carry(q0, k0, dl[k], dev(t[f"v{k + 1}"]), scores, first=k == 0, keep=k + 1 < chain)
        torch.cuda.synchronize()
        assert lb.lisa_kernel_launches() - n0 == (9 if k == 0 else 7)
        assert lb.lisa_check() == lb.OK
        ref = oracle.prefill_rows(f64(t["q0"]), f64(t["k0"]), f64(t[f"v{k + 1}"]), ol[:k + 1], rb, ri)
        assert_close(got[B - 1, torch.from_numpy(ri).long().cuda()].float().cpu().numpy(), ref, "bf16", "concatenating integrate, two waves, layer %d" % (k + 1))


def test_carried_scores_several_waves_from_device_and_host_memory():
    """B = 4, N = 1600: carried scores from device memory are one wave on the caller's stream whatever the prompt's size; the host-memory call
    goes strip by strip on several streams, brings q0, k0, v in and takes o out.  Both must give bit-identical outputs (same kernels on the same data),
    and sampled rows (first and last tile, 32 random rows per sequence) must match the oracle at every depth.  The recomputing calls, whose planes
    exceed one wave's budget, are several waves from either memory."""
    B, N, Hq, Hkv, chain = 4, 1600, 32, 8, 2
    t = link_inputs(B, N, Hq, Hkv, chain, 64, "relu", 2, 21, 43, False)
    dl, ol = make_links(t, chain, "relu")
    rng = np.random.default_rng(1)
    rb, ri = [], []
    for b in range(B):
        rows = np.concatenate([np.arange(128), np.arange(N - 128, N), rng.integers(128, N - 128, 32)])
        rb.append(np.full(rows.shape, b)); ri.append(rows)
    rb, ri = np.concatenate(rb).astype(np.int32), np.concatenate(ri).astype(np.int32)
    scores_d = torch.empty(lb.lisa_prefill_scores_bytes(B, N, Hq), dtype=torch.uint8, device="cuda")
    scores_h = torch.empty_like(scores_d)   # device memory too: the scores of the host-memory calls
    pin = {k: v.pin_memory() for k, v in t.items()}
    q0, k0 = dev(t["q0"]), dev(t["k0"])
    for k in range(chain):
        first, keep = k == 0, k + 1 < chain
        got = lb.lisa_attn_shared_prefill_carry(q0, k0, dl[k], dev(t[f"v{k + 1}"]), scores_d, first=first, keep=keep)
        hl = lb.Link(pin[f"qp{k + 1}"], pin[f"kp{k + 1}"], pin[f"w1_{k + 1}"], pin[f"w2_{k + 1}"], act=lb.ACT_RELU)
        out_h = torch.empty_like(t["q0"]).pin_memory()
        arena = torch.empty(lb.lisa_carry_host_arena_bytes(pin["q0"], pin["k0"], hl, pin[f"v{k + 1}"], out_h, scores_h, first=first),
                            dtype=torch.uint8, device="cuda")
        lb.lisa_attn_shared_prefill_carry_host(pin["q0"], pin["k0"], hl, pin[f"v{k + 1}"], out_h, scores_h, arena, first=first, keep=keep)
        torch.cuda.synchronize()
        assert lb.lisa_check() == lb.OK
        assert torch.equal(out_h, got.cpu())
        ref = oracle.prefill_rows(f64(t["q0"]), f64(t["k0"]), f64(t[f"v{k + 1}"]), ol[:k + 1], rb, ri)
        sel = got[torch.from_numpy(rb).long().cuda(), torch.from_numpy(ri).long().cuda()].float().cpu().numpy()
        assert_close(sel, ref, "bf16", "carried scores, whole prompt and strips, layer %d" % (k + 1))
    # the recomputing call at depth 2 through the host-memory entry point (inputs and output streamed per wave as well)
    hlinks = [lb.Link(pin[f"qp{j}"], pin[f"kp{j}"], pin[f"w1_{j}"], pin[f"w2_{j}"], act=lb.ACT_RELU) for j in (1, 2)]
    out_h = torch.empty_like(t["q0"]).pin_memory()
    arena = torch.empty(lb.lisa_host_arena_bytes(pin["q0"], pin["k0"], hlinks, pin["v2"], out_h), dtype=torch.uint8, device="cuda")
    lb.lisa_attn_shared_prefill_host(pin["q0"], pin["k0"], hlinks, pin["v2"], out_h, arena)
    got2 = lb.lisa_attn_shared_prefill(q0, k0, dl, dev(t["v2"]))
    torch.cuda.synchronize()
    assert torch.equal(out_h, got2.cpu())
    sel = got2[torch.from_numpy(rb).long().cuda(), torch.from_numpy(ri).long().cuda()].float().cpu().numpy()
    assert_close(sel, ref, "bf16", "recomputed in several waves, depth 2")
    assert lb.lisa_check() == lb.OK


@pytest.mark.parametrize("N", [1, 63, 64, 65, 127, 128, 129, 255, 256, 257, 383])
def test_carried_scores_at_tile_boundaries(N):
    """Prompt lengths on and around the 64-key and 128-row tile sizes, three sequences, GQA: two carried layers against the
    oracle, and the second one against the recomputing call of the same depth (the two differ only in where the first
    layer's scores were rounded to fp16)."""
    B, Hq, Hkv, chain = 3, 32, 8, 2
    t = link_inputs(B, N, Hq, Hkv, chain, 64, "relu", 2, 21, 47, True)
    dl, ol = make_links(t, chain, "relu", lb.INTEGRATE_ADD, 2, True)
    scores = torch.full((lb.lisa_prefill_scores_bytes(B, N, Hq),), 0xFF, dtype=torch.uint8, device="cuda")
    q0, k0 = dev(t["q0"]), dev(t["k0"])
    for k in range(chain):
        got = lb.lisa_attn_shared_prefill_carry(q0, k0, dl[k], dev(t[f"v{k + 1}"]), scores, first=k == 0, keep=k + 1 < chain)
        torch.cuda.synchronize()
        assert lb.lisa_check() == lb.OK
        ref = oracle.prefill_full(f64(t["q0"]), f64(t["k0"]), f64(t[f"v{k + 1}"]), ol[:k + 1])
        assert_close(got.float().cpu().numpy(), ref, "bf16", "carried scores, N=%d, layer %d" % (N, k + 1))
    rec = lb.lisa_attn_shared_prefill(q0, k0, dl, dev(t["v2"]))
    torch.cuda.synchronize()
    assert_close(got.float().cpu().numpy(), rec.float().cpu().numpy().astype(np.float64), "bf16", "carried against recomputed, N=%d" % N)


def test_carried_scores_single_layer_keeps_nothing():
    """A chain of one layer through the carried call (first and last at once) equals the recomputing call bit for bit: the
    same kernels run on the same data, only the plane lives in the caller's buffer."""
    B, N, Hq, Hkv = 2, 300, 32, 8
    t = link_inputs(B, N, Hq, Hkv, 1, 64, "silu", 2, 21, 53, False)
    dl, ol = make_links(t, 1, "silu")
    q0, k0, v = dev(t["q0"]), dev(t["k0"]), dev(t["v1"])
    scores = torch.empty(lb.lisa_prefill_scores_bytes(B, N, Hq), dtype=torch.uint8, device="cuda")
    got = lb.lisa_attn_shared_prefill_carry(q0, k0, dl[0], v, scores, first=True, keep=False)
    rec = lb.lisa_attn_shared_prefill(q0, k0, dl, v)
    torch.cuda.synchronize()
    assert lb.lisa_check() == lb.OK
    assert torch.equal(got, rec)
    ref = oracle.prefill_full(f64(t["q0"]), f64(t["k0"]), f64(t["v1"]), ol)
    assert_close(got.float().cpu().numpy(), ref, "bf16", "carried call, single layer")


def test_small_prompt_chain_replayed_from_a_graph():
    """A prompt whose kernels are launched as a programmatic chain, the packing among them: captured and replayed, the results are those of the
    plain calls."""
    B, N, Hkv, chain = 1, 200, 8, 2
    w = synth.Workload("graph", "bf16", B, N, 32, Hkv, 128, 21, 64, "relu", chain)
    t = synth.prefill_inputs(w, 12)
    dl, _ = make_links(t, chain, "relu")
    q0, k0 = dev(t["q0"]), dev(t["k0"])
    vs = [dev(t[f"v{k}"]) for k in range(1, chain + 1)]
    outs = [torch.zeros_like(q0) for _ in range(chain)]
    scores = torch.empty(lb.lisa_prefill_scores_bytes(B, N, 32), dtype=torch.uint8, device="cuda")
    ws = lb.prefill_carry_workspace(q0, k0, dl[0], vs[0], outs[0], scores)

    def layers():
        for k in range(chain):
            lb.lisa_attn_shared_prefill_carry(q0, k0, dl[k], vs[k], scores, first=k == 0, keep=k + 1 < chain, out=outs[k], workspace=ws)
    layers()
    torch.cuda.synchronize()
    ref = [o.clone() for o in outs]
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        layers()
    for o in outs:
        o.zero_()
    g.replay()
    g.replay()
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(outs, ref)) and lb.lisa_check() == lb.OK


@pytest.mark.parametrize("B,N,Hq,Hkv,m,act,bias", [
    (3, 385, 32, 8, 64, "relu", True),     # 32 -> 64 -> 32 above one wave of CTAs; odd row count: a tile's second row lies past the prompt
    (3, 447, 32, 32, 1, "silu", True),     # one hidden unit in a padded k-step
    (3, 385, 32, 8, 33, "none", False),    # 48 hidden units of the MMAs, the last 15 zero
    (3, 512, 32, 32, 112, "silu", True),   # remainder of the 32-unit chunks
    (3, 385, 32, 8, 129, "relu", True),    # the second warpgroup of a tile has one k-step
    (3, 386, 40, 40, 129, "relu", True)])  # 40 heads over two warpgroups: three groups and two
def test_single_links_of_several_waves_take_the_link_kernel(B, N, Hq, Hkv, m, act, bias):
    """One-link calls of more than one wave of CTAs: recomputed, and as two layers that carry the scores."""
    t = link_inputs(B, N, Hq, Hkv, 2, m, act, 2, 21, 41, bias)
    dl, ol = make_links(t, 2, act, lb.INTEGRATE_ADD, 2, bias)
    q0, k0 = dev(t["q0"]), dev(t["k0"])
    ref = [oracle.prefill_full(f64(t["q0"]), f64(t["k0"]), f64(t[f"v{k + 1}"]), ol[:k + 1]) for k in range(2)]
    got = lb.lisa_attn_shared_prefill(q0, k0, dl[:1], dev(t["v1"]))
    assert_close(got.float().cpu().numpy(), ref[0], "bf16", "one link, recomputed")
    scores = torch.full((lb.lisa_prefill_scores_bytes(B, N, Hq),), 0xFF, dtype=torch.uint8, device="cuda")
    for k in range(2):
        got = lb.lisa_attn_shared_prefill_carry(q0, k0, dl[k], dev(t[f"v{k + 1}"]), scores, first=k == 0, keep=k == 0)
        assert_close(got.float().cpu().numpy(), ref[k], "bf16", "one link a call, layer %d" % (k + 1))
    assert lb.lisa_check() == lb.OK


@pytest.mark.parametrize("N", [1, 64, 65, 129, 193, 384])
@pytest.mark.parametrize("form", ["anchor", "plane", "carry"])
def test_attention_whose_maxima_keep_growing(N, form):
    """Scores that rise along the keys by 3 every 16, and fall by 2 every 40 on top: nearly every tile moves the reference maximum of its rows
    (the accumulator is rescaled, and one warpgroup's sum meets a reference the other has set).  Scores up to 72 are rounded where the kernels
    round them: Q.K (or Q'.K') in fp32 from bf16 products, exact here; so the stated bar holds."""
    j = torch.arange(N)
    a = (j // 16 * 3 - j % 40 // 20 * 2).float()                       # whole numbers below 256: exact in bf16
    v = synth.as_dtype(synth.normal("v", (1, N, 32, 128), 5), "bf16")
    r = 16
    if form == "anchor":
        q, k = torch.zeros(1, N, 32, 128), torch.zeros(1, N, 32, 128)
        q[..., 0], k[..., 0] = 1.0, a[None, :, None]
        scale = 128 ** -0.5
        q = q * 8.0                                                    # score = a / sqrt(2)
        s = (8.0 * scale * a).double()
        got = lb.lisa_attn_anchor(dev(q.bfloat16()), dev(k.bfloat16()), dev(v))
    else:
        z = synth.as_dtype(synth.normal("q", (1, N, 32, 128), 6), "bf16")
        qp, kp = torch.zeros(1, N, 32, r), torch.zeros(1, N, 32, r)
        qp[..., 0], kp[..., 0] = 4.0, a[None, :, None]                 # score = a, with an aligner of zero weights
        s = a.double()
        link = lb.Link(dev(qp.bfloat16()), dev(kp.bfloat16()), torch.zeros(32, 64, dtype=torch.bfloat16, device="cuda"),
                       torch.zeros(64, 32, dtype=torch.bfloat16, device="cuda"))
        if form == "plane":
            got = lb.lisa_attn_shared_prefill(dev(z), dev(z), [link], dev(v))
        else:
            scores = torch.empty(lb.lisa_prefill_scores_bytes(1, N, 32), dtype=torch.uint8, device="cuda")
            got = lb.lisa_attn_shared_prefill_carry(dev(z), dev(z), link, dev(v), scores, first=True, keep=True)
    torch.cuda.synchronize()
    assert lb.lisa_check() == lb.OK
    p = torch.softmax(s[None, :].expand(N, N).masked_fill(torch.ones(N, N, dtype=torch.bool).triu(1), float("-inf")), -1)
    ref = torch.einsum("ij,bjhd->bihd", p, v.double())
    assert_close(got.float().cpu().numpy(), ref.numpy(), "bf16", form)


CHAIN_FORMS = [(32, lb.INTEGRATE_ADD), (40, lb.INTEGRATE_ADD), (32, lb.INTEGRATE_CONCAT)]


# (4500 tokens: 1152 CTAs of a head-partitioned kernel, nearly four rounds, in one programmatic chain)
@pytest.mark.parametrize("Hq,integrate,N", [(*form, N) for form in CHAIN_FORMS for N in (50, 197, 1300)] + [(32, lb.INTEGRATE_ADD, 4500)])
def test_a_programmatic_chain_equals_its_kernels_one_by_one(Hq, integrate, N):
    """A carried chain of two layers, a fresh scores buffer and workspace for each of three inputs, called back to back: every output as with the
    per-kernel timing on, which takes the chain apart (packing first, every kernel behind the one before)."""
    m, h_in = 64, Hq * (2 if integrate == lb.INTEGRATE_CONCAT else 1)

    def inputs(seed):
        n = lambda name, *shape: dev(synth.as_dtype(synth.normal(name, shape, seed), "bf16"))  # noqa: E731
        w = lambda name, *shape: dev(synth.as_dtype(synth.normal(name, shape, seed, std=shape[0] ** -0.5), "bf16"))  # noqa: E731
        return n("q", 1, N, Hq, 128), n("k", 1, N, Hq, 128), [
            (n("v%d" % k, 1, N, Hq, 128), lb.Link(n("qp%d" % k, 1, N, Hq, 21), n("kp%d" % k, 1, N, Hq, 21), w("w1%d" % k, h_in, m), w("w2%d" % k, m, Hq),
                                                  integrate=integrate)) for k in range(2)]

    def run(all_in):
        outs = []
        for q, k, layers in all_in:
            scores = torch.empty(lb.lisa_prefill_scores_bytes(1, N, Hq), dtype=torch.uint8, device="cuda")
            for i, (v, link) in enumerate(layers):
                outs.append(lb.lisa_attn_shared_prefill_carry(q, k, link, v, scores, first=i == 0, keep=i == 0))
        torch.cuda.synchronize()
        assert lb.lisa_check() == lb.OK
        return outs

    all_in = [inputs(s) for s in (1, 2, 3)]
    lb.lisa_prefill_phase_timing(True)
    try:
        ref = run(all_in)
    finally:
        lb.lisa_prefill_phase_timing(False)
    for _ in range(3):
        assert all(torch.equal(x, y) for x, y in zip(run(all_in), ref))


@pytest.mark.parametrize("by", ["project", "copy"])
@pytest.mark.parametrize("Hq,integrate,N", [(32, lb.INTEGRATE_ADD, 197), (32, lb.INTEGRATE_CONCAT, 333), (40, lb.INTEGRATE_ADD, 333)])
def test_inputs_rewritten_right_before_a_chained_call(Hq, integrate, N, by):
    """A serving loop's buffers: Q', K', V (a projection, or copies), the cache append and the aligner's weights are written into the same
    tensors for every layer and prompt, by the kernels right in front of the carried call, first layer and later ones, one workspace for all.
    Every output as with the per-kernel timing on, which takes the chain apart."""
    m, h_in, r, passes = 64, Hq * (2 if integrate == lb.INTEGRATE_CONCAT else 1), 21, 6
    g = torch.Generator(device="cuda").manual_seed(N)
    n = lambda *shape, std=1.0: torch.randn(shape, generator=g, device="cuda").mul_(std).bfloat16()  # noqa: E731
    q0, k0, h = n(1, N, Hq, 128), n(1, N, Hq, 128), n(1, N, 256)
    w_in = [n(256, Hq * (2 * r + 128), std=256 ** -0.5) for _ in range(passes)]
    new = [(n(1, N, Hq, r), n(1, N, Hq, r), n(1, N, Hq, 128)) for _ in range(passes)]
    ffn = [(n(h_in, m, std=h_in ** -0.5), n(m, Hq, std=m ** -0.5)) for _ in range(passes)]
    qp, kp, v = (torch.zeros_like(x) for x in new[0])
    w1, w2 = (torch.zeros_like(x) for x in ffn[0])
    cache = lb.KVCacheLayer(lb.CACHE_SHARED, 1, Hq, (N + 71) // 8 * 8, 128, r, dtype=torch.bfloat16)
    scores = torch.empty(lb.lisa_prefill_scores_bytes(1, N, Hq), dtype=torch.uint8, device="cuda")
    link = lb.Link(qp, kp, w1, w2, integrate=integrate)
    ws = lb.prefill_carry_workspace(q0, k0, link, v, torch.empty_like(q0), scores)

    def run():
        outs = [torch.empty_like(q0) for _ in range(passes)]
        for i in range(passes):
            if by == "project":
                lb.lisa_project(h, w_in[i], [qp, kp, v])
            else:
                for dst, src in zip((v, kp, qp), reversed(new[i])):
                    dst.copy_(src)
            if i % 2:
                lb.lisa_kvcache_append(cache, kp, v)
            for dst, src in zip((w2, w1), reversed(ffn[i])):
                dst.copy_(src)
            if i % 3 == 2:   # the weights' copies are not the last kernels in front of the call
                lb.lisa_kvcache_append(cache, kp, v)
            lb.lisa_attn_shared_prefill_carry(q0, k0, link, v, scores, first=i % 3 == 0, keep=i % 3 < 2, out=outs[i], workspace=ws)
        torch.cuda.synchronize()
        assert lb.lisa_check() == lb.OK
        return outs

    lb.lisa_prefill_phase_timing(True)
    try:
        ref = run()
    finally:
        lb.lisa_prefill_phase_timing(False)
    assert not any(torch.equal(ref[i], ref[i + 1]) for i in range(passes - 1))
    for _ in range(5):
        assert all(torch.equal(x, y) for x, y in zip(run(), ref))


@pytest.mark.parametrize("r", [1, 15, 16, 17, 31, 32])
def test_low_ranks_at_the_edges_of_their_padding(r):
    """Q' and K' are packed into rows of 32, of which whole groups of 16 are multiplied: with an emitted difference (chain of two) and without."""
    run_tc_shared(1, 200, 8, 1, "relu", seed=r, r=r)
    run_tc_shared(2, 130, 32, 2, "silu", seed=r, r=r)


@pytest.mark.parametrize("r,Hkv", [(21, 32), (21, 4), (20, 8), (1, 1), (7, 2), (32, 32)])
def test_low_ranks_are_packed_alike_wherever_their_rows_start(r, Hkv):
    """Rows of Q' and K' that start on 16, 4 and 2 bytes, heads with a stride of their own, a row of values that is no whole number of
    16-byte units: the outputs of the dense tensors, bit for bit.  N is no multiple of the eight positions a CTA packs."""
    w = synth.Workload("tc_pack", "bf16", 2, 203, 32, Hkv, 128, r, 64, "relu", 1)
    t = synth.prefill_inputs(w, r)
    q0, k0, v, w1, w2 = (dev(t[n]) for n in ("q0", "k0", "v1", "w1_1", "w2_1"))

    def run(qp, kp):
        out = lb.lisa_attn_shared_prefill(q0, k0, [lb.Link(qp, kp, w1, w2, act=lb.ACT_RELU)], v)
        torch.cuda.synchronize()
        assert lb.lisa_check() == lb.OK
        return out

    def strided(x, more, head):
        B, N, H, n = x.shape
        row = H * head + more
        y = torch.zeros(B * N * row + 8, dtype=x.dtype, device="cuda").as_strided((B, N, H, n), (N * row, row, head, 1))
        return y.copy_(x)

    qp, kp = dev(t["qp1"]), dev(t["kp1"])
    ref = run(qp, kp)
    for more, head in ((8, r), (2, r), (1, r), (0, r + 3)):
        assert torch.equal(run(strided(qp, more, head), strided(kp, more, head)), ref), (more, head)


@pytest.mark.parametrize("B,N,Hq,Hkv", [(6, 4096, 32, 32), (3, 5000, 40, 40), (5, 7000, 32, 8)])
def test_attention_whose_keys_and_values_exceed_l2(B, N, Hq, Hkv):
    """Past 63 MB of K and V the (batch, head) pairs are handed out in groups (whole batches, then parts of one): every pair and query tile is computed
    once, whatever the order.  The heads of a few KV heads at a time, of all sequences, whose K and V fit: one group, heads and sequences side by side;
    the same bytes.  Rows of the first and last tiles of the last sequence, all heads of it, are the oracle's."""
    g = torch.Generator(device="cuda").manual_seed(B)
    q, k, v = (torch.randn((B, N, h, 128), generator=g, device="cuda", dtype=torch.bfloat16) for h in (Hq, Hkv, Hkv))
    got = torch.full_like(q, float("nan"))
    lb.lisa_attn_anchor(q, k, v, out=got)
    G, at_once = Hq // Hkv, (63 << 20) // (B * N * 512)
    assert 1 <= at_once < Hkv
    for a in range(0, Hkv, at_once):
        b = min(a + at_once, Hkv)
        part = lb.lisa_attn_anchor(q[:, :, a * G:b * G], k[:, :, a:b], v[:, :, a:b])
        assert torch.equal(part, got[:, :, a * G:b * G]), (a, b)
    assert lb.lisa_check() == lb.OK
    rows = np.array([0, 1, 63, 64, 127, 128, N - 130, N - 65, N - 1], dtype=np.int32)
    ref = oracle.prefill_rows(*(f64(x[B - 1:].cpu()) for x in (q, k, v)), [], np.zeros_like(rows), rows)
    assert_close(got[B - 1, torch.from_numpy(rows).long().cuda()].float().cpu().numpy(), ref, "bf16", "rows of the last sequence")
