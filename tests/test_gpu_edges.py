"""Edges of the tiles and dispatch rules of the kernels: sizes around a tile, a warp, a cluster, the switch from
one kernel to another, and the smallest ones, against the oracle or a 64-bit product.

Tolerances.  Activations travel as bf16 hi + lo: x - (hi + lo) is at most 2^-17 |x|; products are accumulated in
fp32 with fewer than 2^5 x 2^3 additions in a row per lane, warp and tile, so an element of X W^T is off by at
most (2^-17 + 2^8 2^-24) sum |x| |w|: 2^-15 of that sum bounds it.  fp32 weights: 2^-17 of the same sum.
Counts, tokens and truncated rows are exact.
"""
import numpy as np
import pytest

import synth
from oracle import adapter as OA
from oracle import sampling as S
from oracle import warp

import harness as H

from test_gpu_adapter import _run, _tiny_ctx
from test_gpu_spd import _lib, lockstep
from test_gpu_truncate import _dev_truncate

F32 = np.float32


@pytest.mark.gpu
@pytest.mark.parametrize("M,N,K,dtype", [
    (1, 1, 8, 1), (2, 15, 24, 1), (3, 17, 32, 1), (8, 147, 40, 1), (5, 149, 1000, 1), (7, 2369, 2048, 1),
    (6, 297, 6144, 1), (6, 297, 6152, 1),          # the last K whose fragments fit shared memory, the first that does not
    (1, 1, 8, 0), (2, 3, 120, 0), (8, 5, 128, 0), (7, 150, 136, 0), (4, 593, 2056, 0),
    (8, 33, 6144, 0), (8, 33, 6152, 0), (3, 64, 16384, 0)])
@pytest.mark.parametrize("noalloc", [False, True])
def test_skinny_gemm_edges(M, N, K, dtype, noalloc):
    import torch
    spd = _lib()
    g = np.random.default_rng(M * 100000 + N * 10 + dtype)
    x = g.standard_normal((M, K)).astype(F32)
    w = (g.standard_normal((N, K)) * 0.05).astype(F32)
    wd = torch.from_numpy(w).cuda()
    if dtype == 1:
        bits = synth.f32_to_bf16_bits(w)
        w, wd = synth.bf16_bits_to_f32(bits), torch.from_numpy(bits.view(np.int16)).cuda()
    y = torch.full((M, N), float("nan"), device="cuda")
    (spd.skinny_gemm_noalloc if noalloc else spd.skinny_gemm)(torch.from_numpy(x).cuda(), wd, y, dtype)
    torch.cuda.synchronize()
    want = x.astype(np.float64) @ w.astype(np.float64).T
    bound = np.abs(x).astype(np.float64) @ np.abs(w).astype(np.float64).T * 2.0 ** (-15 if dtype else -17)
    got = y.cpu().numpy()
    assert np.isfinite(got).all() and (np.abs(got - want) <= bound).all()
    assert spd.skinny_gemm_status(noalloc) == 0


@pytest.mark.gpu
@pytest.mark.parametrize("B,gamma,V", [(1, 0, 1), (3, 1, 31), (2, 9, 1024), (20, 7, 4099), (75, 2, 8200), (149, 17, 700), (1, 5, 40000),
                                       (2, 40, 6144), (2, 33, 6145), (5, 3, 16384), (5, 3, 16385), (40, 1, 16390), (3, 4, 33),
                                       (8, 9, 1999), (8, 7, 4000), (9, 8, 4097), (10, 8, 8000), (18, 1, 16400), (7, 8, 4096)])
def test_rejection_rule_edges(B, gamma, V):
    """Every cluster width, more rows than are taken together when greedy, vocabularies around a warp's piece."""
    import torch
    spd = _lib()
    tl, dl = synth.microbench_logits(B, max(gamma, 1), V, 0.3)
    p = S.softmax_t(np.ascontiguousarray(tl[:, :gamma + 1]), 1.0)
    q = S.softmax_t(np.ascontiguousarray(dl[:, :gamma]), 1.0) if gamma else np.zeros((B, 0, V), F32)
    for greedy in (False, True):
        ids = (p[:, :gamma] if greedy else q).argmax(-1).astype(np.int32).reshape(B, gamma)
        if greedy and gamma > 8:
            ids[::2, 8] = (ids[::2, 8] + 1) % V        # a mismatch in the second group of rows
        u = synth.uniforms(9, f"edge.{B}.{V}", (B, gamma + 1))
        want_a, want_n = S.reject_sample_batch(p, q, ids, u, greedy)
        a, n = (torch.full((B,), -7, dtype=torch.int32, device="cuda") for _ in range(2))
        dev = [torch.from_numpy(np.ascontiguousarray(t)).cuda() if t.size else torch.zeros(1, device="cuda").to(torch.int32 if t is ids else torch.float32)
               for t in (p, q, ids, u)]
        spd.reject_sample(*dev, gamma, greedy, a, n)
        assert np.array_equal(a.cpu().numpy(), want_a) and np.array_equal(n.cpu().numpy(), want_n)


@pytest.mark.gpu
@pytest.mark.parametrize("V", [1023, 1025, 32768, 53700, 56500])     # the last two: many and few digit bins fit beside the row
def test_truncation_edges(V):
    spd = _lib()
    g = np.random.default_rng(V)
    raw = np.floor(g.standard_exponential((3, V)) * 6).astype(F32)
    raw[:, V // 2] += 1
    rows = (raw / raw.sum(axis=1, keepdims=True)).astype(F32)
    rows[1] = S.softmax_t(g.standard_normal((1, V)).astype(F32) * 3, 1.0)[0]
    for top_k, top_p in [(1, 1.0), (V - 1, 0.5), (50, 0.9), (0, 0.9999)]:
        want = warp.warp_rows(rows, top_k, top_p)
        assert np.array_equal(_dev_truncate(spd, rows, top_k, top_p).view(np.uint32), want.view(np.uint32)), (top_k, top_p)


@pytest.mark.gpu
@pytest.mark.parametrize("m,d_in,d_hid,d_out", [(15, 64, 136, 128), (17, 72, 264, 257), (31, 128, 120, 1), (129, 200, 512, 130),
                                               (257, 256, 256, 384), (513, 1024, 2312, 256)])
def test_image_adapter_edges(m, d_in, d_hid, d_out):
    """Row counts around the activation tiles (multiples of 16, 32 and 256), ragged widths, one and several K blocks;
    the bound is the one of the adapter's own test."""
    _lib()
    gpu = _tiny_ctx()
    feats = synth.vision_features(2, m, d_in)
    w1, w2 = synth.adapter_mlp(1, "target", d_in, d_hid, d_out, std=0.05)
    want = OA.image_adapter(feats, synth.bf16_bits_to_f32(w1), synth.bf16_bits_to_f32(w2))
    got = _run(gpu, feats, w1, w2, False)
    assert np.isfinite(got).all() and (np.abs(got - want) <= 1e-4 + 1e-4 * np.abs(want)).all()
    gpu.close()


@pytest.mark.gpu
@pytest.mark.parametrize("n_image,n_prompt", [(0, 1), (0, 63), (1, 64), (64, 65), (100, 157)])
@pytest.mark.parametrize("d_draft,heads", [(128, 2), (256, 2)])
def test_prompt_lengths_around_the_attention_tiles(n_image, n_prompt, d_draft, heads):
    """Prefill attention (64-row tiles, heads of 64 and 128) in lock-step with the oracle; the logit bound is that of
    the other small bf16 models."""
    t = synth.ModelCfg(1, 256, 2, 264, 1000, False, dtype="bf16")
    d = synth.ModelCfg(2, d_draft, heads, 344, 1000, True, dtype="bf16")
    wl = synth.Workload("edge", t, d, n_image, n_prompt, 4, 16)
    assert lockstep(wl, False, 1.0, 2, 2e-2, std=0.08)["blocks"] == 2


@pytest.mark.gpu
def test_a_prompt_is_summed_in_the_same_order_whatever_came_before_it():
    """540 rows of a 256-wide model: a length at which the room for K slices depends on the rows it is taken from.
    Logits bit for bit on a fresh context, behind a longer prompt, and on a fork of the context that had it."""
    _lib()
    t = synth.ModelCfg(1, 256, 2, 264, 1000, False, dtype="bf16")
    d = synth.ModelCfg(1, 128, 2, 344, 1000, True, dtype="bf16")
    wl = synth.Workload("order", t, d, 0, 540, 4, 16)
    tw, dw = H.build_weights(wl, 0.08)
    gpu = H.make_gpu(wl, tw, dw, 2100, 1.0, True)
    ids = synth.prompt_ids(wl)
    longer = np.resize(ids, 2048).astype(np.int32)

    def logits(ctx):
        ctx.prefill(None, ids)
        return ctx.get_logits(1).copy()

    fresh = logits(gpu)
    gpu.prefill(None, longer)
    again, other = logits(gpu), gpu.fork()
    forked = logits(other)
    assert np.array_equal(fresh.view(np.uint32), again.view(np.uint32))
    assert np.array_equal(fresh.view(np.uint32), forked.view(np.uint32))
    other.close()
    gpu.close()


@pytest.mark.gpu
@pytest.mark.parametrize("V", [64, 1000, 4100, 32000])
def test_draws_from_rows_that_are_no_distribution(V):
    """Rows of NaN, of infinity and without any mass give a token of the vocabulary, in one CTA and across clusters.
    A NaN counts 2^63, so an even number of them adds up to no mass (modulo 2^64): then the largest weight, lowest
    index, of the entries that are numbers, and 0 if there is none."""
    import torch
    spd = _lib()
    nan, inf = np.nan, np.inf
    tiny = np.full(V, nan, F32)
    tiny[[7, V - 3]] = [1e-12, 2e-12]
    one = np.zeros(V, F32)
    one[V - 5] = inf
    flat = np.full(V, 1.0 / V, F32)
    half = np.zeros(V, F32)            # target 1/2 of the draft everywhere: nothing is left after a rejection
    half[: V // 2] = 1.0 / V
    # (target row under test, draft row, u of the accept test, accepted, next)
    rows = [(np.full(V, nan, F32), flat, 0.5, 1, 0), (tiny, flat, 0.5, 1, V - 3), (one, flat, 0.5, 1, V - 5), (half, 2 * half, 0.75, 0, 0)]
    p = np.stack([np.stack([flat if a else t, t]) for t, _, _, a, _ in rows])
    q = np.stack([d[None] for _, d, _, _, _ in rows])
    u = np.array([[x, 0.25] for _, _, x, _, _ in rows], F32)
    ids = np.zeros((len(rows), 1), np.int32)
    a, n = (torch.full((len(rows),), -7, dtype=torch.int32, device="cuda") for _ in range(2))
    dev = [torch.from_numpy(x).cuda() for x in (p, q, ids, u)]
    spd.reject_sample(*dev, 1, False, a, n)
    assert a.cpu().tolist() == [r[3] for r in rows] and n.cpu().tolist() == [r[4] for r in rows]
    greedy = np.stack([np.full((2, V), x, F32) for x in (nan, -inf)] + [np.stack([one, one])])
    ids = np.array([[0], [0], [V - 5]], np.int32)
    spd.reject_sample(torch.from_numpy(greedy).cuda(), None, torch.from_numpy(ids).cuda(), None, 1, True, a[:3], n[:3])
    assert a[:3].cpu().tolist() == [1, 1, 1] and n[:3].cpu().tolist() == [0, 0, V - 5]
    ties = np.zeros((3, V), F32)                       # equal values in several pieces, zeros of both signs
    ties[0, [V // 2, V // 2 + 31, V - 1]] = 2.0
    ties[1, ::2] = -0.0
    ties[2] = -3.0
    ties[2, [V // 3, V - 2]] = -0.0
    ids = ties.argmax(-1).astype(np.int32)[:2][None]
    spd.reject_sample(torch.from_numpy(ties[None]).cuda(), None, torch.from_numpy(ids).cuda(), None, 2, True, a[:1], n[:1])
    assert (int(a[0]), int(n[0])) == (2, V // 3)
    trunc = np.stack([np.where(np.arange(V) % 3 == 1, F32(nan), flat), np.where(np.arange(V) % 2 == 0, -flat, flat)]).astype(F32)
    want = warp.warp_rows(np.where(trunc > 0, trunc, F32(0)), 20, 0.9)
    assert np.array_equal(_dev_truncate(spd, trunc, 20, 0.9).view(np.uint32), want.view(np.uint32))


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
def test_a_step_whose_logits_are_nan_yields_a_token_of_the_vocabulary(dtype):
    """NaN image rows make every logit of the target NaN: the first token and the one a verify step emits are 0."""
    _lib()
    t = synth.ModelCfg(2, 256, 4, 688, 1024, False, dtype=dtype)
    d = synth.ModelCfg(1, 128, 2, 344, 1024, False, dtype=dtype)
    wl = synth.Workload("nan", t, d, 16, 16, 4, 32)
    tw, dw = H.build_weights(wl, 0.1)
    gpu = H.make_gpu(wl, tw, dw, 96, 1.0, False)
    img, ids = synth.image_embeds(wl), synth.prompt_ids(wl)
    u = synth.uniforms(5, "nan", 8)
    assert gpu.prefill(np.full_like(img, np.nan), ids, u0=0.5) == 0
    gpu.draft(2, u[:2])
    assert gpu.verify(2, u[2:5])[1] == 0
    assert np.isnan(gpu.get_logits(3)).all()
    gpu.draft(2, u[:2])                     # the next step takes the emitted token as it is
    gpu.verify(2, u[2:5])
    gpu.close()


def _small_bf16_on_a_stream(stream, greedy=True):
    spd = _lib()
    t = synth.ModelCfg(1, 256, 4, 344, 1024, False, dtype="bf16")
    d = synth.ModelCfg(1, 128, 2, 344, 1024, False, dtype="bf16")
    wl = synth.Workload("stream", t, d, 0, 16, 4, 16)
    tw, dw = H.build_weights(wl, 0.15)
    return spd, wl, spd.Spd(t, d, tw.stored, dw.stored, 96, 7, 1.0, greedy, stream=stream.cuda_stream)


def _refused_while_capturing(spd, stream, call):
    import torch
    x = torch.zeros(8, device="cuda")
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        graph = torch.cuda.CUDAGraph()
        graph.capture_begin()
        try:
            x.add_(1)
            with pytest.raises(spd.SpdError) as e:
                call()
        finally:
            graph.capture_end()
    assert e.value.status == spd.SPD_ECUDA


@pytest.mark.gpu
def test_rollback_is_refused_while_the_stream_is_being_captured():
    """The host's bound on the sequence length must not follow a rollback that may never run."""
    import torch
    stream = torch.cuda.Stream()
    spd, wl, gpu = _small_bf16_on_a_stream(stream)
    ids = synth.prompt_ids(wl)
    first = gpu.prefill(None, ids)
    want, _ = gpu.generate(8, 4)
    at = gpu.get_state()
    _refused_while_capturing(spd, stream, lambda: gpu.rollback(len(ids), int(ids[-1]), first))
    assert gpu.get_state() == at
    gpu.rollback(len(ids), int(ids[-1]), first)
    got, _ = gpu.generate(8, 4)
    assert np.array_equal(got, want)
    gpu.close()


@pytest.mark.gpu
def test_batched_steps_are_refused_while_the_stream_is_being_captured():
    """... neither on a batch that has never run, whose descriptors would not reach the device, nor on a used one."""
    import torch
    stream = torch.cuda.Stream()
    spd, wl, gpu = _small_bf16_on_a_stream(stream)
    ids = synth.prompt_ids(wl)
    first = gpu.prefill(None, ids)
    want, _ = gpu.generate(16, 3)
    other = gpu.fork()
    for c in (gpu, other):
        c.prefill(None, ids)
    bt = spd.SpdBatch([gpu, other])
    got = [[first], [first]]
    for _ in range(3):
        _refused_while_capturing(spd, stream, lambda: bt.draft(3, read_ids=False))
        d = bt.draft(3)
        _refused_while_capturing(spd, stream, lambda: bt.verify(3, read=False))
        a, n = bt.verify(3)
        for k in range(2):
            got[k] += [int(x) for x in d[k][: a[k]]] + [int(n[k])]
    for k in range(2):
        m = min(len(got[k]), 16)
        assert got[k][:m] == want[:m].tolist()
    bt.close()
    other.close()
    gpu.close()


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
def test_draft_logits_of_every_step_are_kept(dtype):
    """gamma = 7: all seven rows, whose softmax is the step's distribution (the same numbers but for the order of
    one sum: 2^-18 of each); what a later call has written over is refused, the rest is unchanged."""
    import torch
    spd = _lib()
    t = synth.ModelCfg(1, 256, 4, 344, 1024, False, dtype=dtype)
    d = synth.ModelCfg(2, 128, 2, 344, 1024, False, dtype=dtype)
    wl = synth.Workload("rows", t, d, 0, 16, 7, 16)
    tw, dw = H.build_weights(wl, 0.1)
    gpu = H.make_gpu(wl, tw, dw, 96, 1.0, False)
    gpu.prefill(None, synth.prompt_ids(wl), u0=0.5)
    u = synth.uniforms(3, "rows", 16)
    probs = torch.zeros(7, 1024, device="cuda")
    gpu.draft(7, u[:7], probs_out=probs)
    rows = gpu.get_draft_logits(7)
    want = probs.cpu().numpy()
    assert (np.abs(S.softmax_t(rows, 1.0) - want) <= 2.0 ** -18 * want + 1e-12).all()
    for branching, left in (([1, 1, 1], 6), ([4], 6), ([2, 2], 6), ([3, 1], 5)):
        gpu.draft_tree(branching, u[:7])
        for refused in range(left + 1, 8):
            with pytest.raises(spd.SpdError) as e:
                gpu.get_draft_logits(refused)
            assert e.value.status == spd.SPD_EINVAL
        assert np.array_equal(gpu.get_draft_logits(left).view(np.uint32), rows[:left].view(np.uint32))
    gpu.close()


@pytest.mark.gpu
def test_threads_that_truncate_rows_of_different_lengths_at_once():
    """The kernels' limit on shared memory belongs to the process: no thread may lower it under another's launch.
    A fresh process, so that the first calls of all threads come together."""
    import subprocess
    import sys
    code = """
import sys, threading
import numpy as np, torch
import paper_2404_08856_b200 as spd
spd.lib(); torch.cuda.init()
sizes = [56500, 53000, 40000, 30000, 20000, 13000, 5000, 54500]
rows = [torch.full((2, V), 1.0 / V, device="cuda") for V in sizes]
outs = [torch.empty_like(r) for r in rows]
torch.cuda.synchronize()
gate, bad = threading.Barrier(len(sizes)), []
def work(i):
    torch.cuda.set_device(0)
    gate.wait()
    for _ in range(50):
        try:
            spd.truncate_probs(rows[i], outs[i], 3, 1.0)
        except Exception as e:
            bad.append((sizes[i], str(e)))
threads = [threading.Thread(target=work, args=(i,)) for i in range(len(sizes))]
[t.start() for t in threads]; [t.join() for t in threads]
torch.cuda.synchronize()
assert not bad, bad[:3]
for V, o in zip(sizes, outs):
    assert (o.cpu().numpy() > 0).sum(1).tolist() == [3, 3] and float(o[0, 0]) > 0, V
print("threads ok")
"""
    import os
    _lib()
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, cwd=root, timeout=200)
    assert r.returncode == 0 and "threads ok" in r.stdout, r.stderr[-2000:]


@pytest.mark.gpu
@pytest.mark.parametrize("dtype,tol", [("fp32", 2e-4), ("bf16", 2e-2)])
def test_models_wider_than_their_vocabulary_and_ffn(dtype, tol):
    """The largest matrix of the target is d_model x d_model, that of the draft its adapter."""
    t = synth.ModelCfg(1, 512, 4, 264, 400, False, dtype=dtype)
    d = synth.ModelCfg(1, 128, 2, 136, 400, False, dtype=dtype)
    wl = synth.Workload("wide", t, d, 8, 16, 4, 16, adapter_in=512)
    assert lockstep(wl, False, 1.0, 2, tol, std=0.08)["blocks"] == 2
