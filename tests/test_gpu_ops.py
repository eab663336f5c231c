"""Kernel-level parity through the C-ABI single-op entry points: the tcgen05 GEMM (all
epilogues, ragged M, both N tile widths), the CUDA-core GEMM, and flash attention
(self / shared-K/V cross, head_dim 64 and 128, ragged tails) against the oracle's fp64
primitives on the same bf16 inputs."""
import os
import subprocess
import sys
import threading

import numpy as np
import pytest
import torch

from oracle import flashbon_oracle as O
from paper_2607_04461_gb300 import flashbon as fb
from paper_2607_04461_gb300 import synth
from _metrics import rel_max

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def model():
    fb.load_library()
    m = fb.Model(synth.TINY, synth.make_weights(synth.TINY))
    yield m
    m.close()


def randn(shape, seed, scale=1.0, dtype=torch.bfloat16):
    g = torch.Generator().manual_seed(seed)
    return (torch.randn(shape, generator=g) * scale).to(dtype).cuda()


def f64(t):
    return t.float().cpu().double().numpy()


GEMM_SHAPES = [
    (300, 256, 128),     # ragged M, BN=128, two K blocks
    (1, 128, 64),        # one row, one K block
    (2500, 384, 192),    # many tiles, BN=128
    (4000, 4608, 256),   # >= one tile per SM at BN=256 (the QKV shape's N)
    (640, 1536, 8960),   # long K (FFN down)
]


@pytest.mark.parametrize("M,N,K", GEMM_SHAPES)
@pytest.mark.parametrize("epi", [0, 1, 2, 3])
def test_gemm_tc(model, M, N, K, epi):
    """Automatic choice: the 2-SM kernel when N % 256 == 0, else the 1-SM kernel."""
    _gemm_case(model, M, N, K, epi, impl=0)


@pytest.mark.parametrize("M,N,K", [(300, 256, 128), (1560, 1536, 1536), (513, 512, 8960)])
@pytest.mark.parametrize("epi", [0, 3])
def test_gemm_tc_1sm_forced(model, M, N, K, epi):
    _gemm_case(model, M, N, K, epi, impl=2)


@pytest.mark.parametrize("M", [1, 129, 256, 257, 1560, 49920])
def test_gemm_tc_2sm_ragged_rows(model, M):
    """Pair tiles of 256 rows: rows of the odd CTA may lie wholly past M."""
    _gemm_case(model, M, 512, 128, 0, impl=0)


@pytest.mark.parametrize("M,N,K", [
    (5, 256, 64),        # fewer rows than the narrowest tile, one K block
    (100, 2304, 192),    # one token tile per feature tile, a ragged last chunk
    (700, 1536, 320),    # narrow tiles, 5 K blocks (both loading warps, uneven)
    (1560, 1536, 128),   # 11 token tiles, the last one partial
    (1560, 4608, 640),   # two rounds
    (2049, 512, 1536),   # one row in the last tile
    (700, 128, 1536),    # every tile half empty
    (3000, 384, 1600),   # the last feature tile half empty
])
@pytest.mark.parametrize("epi", [0, 1, 2, 3])
def test_gemm_2sm_tile_widths(model, M, N, K, epi):
    """The 2-SM kernel fits its tiles' token width to M: every width class, ragged last
    tiles and chunks, against the fp64 product; rows past M stay untouched."""
    A = randn((M, K), 71)
    W = randn((N, K), 72, scale=K ** -0.5)
    bias, gate = randn((N,), 73, dtype=torch.float32), randn((N,), 74, dtype=torch.float32)
    resid = randn((M, N), 75, dtype=torch.float32) if epi >= 2 else None
    base = randn((M, N), 76, dtype=torch.float32) if epi == 3 else None
    out = torch.full((M + 32, N), 7.0, dtype=torch.float32 if epi >= 2 else torch.bfloat16,
                     device="cuda")
    delta = torch.full((M + 32, N), 7.0, dtype=torch.bfloat16, device="cuda")
    fb.fb_op_gemm(model.handle, M, N, K, A, W, bias, epi, out, resid,
                  gate if epi >= 2 else None, base, delta if epi == 3 else None, 3)
    torch.cuda.synchronize()
    assert torch.all(out[M:] == 7.0) and torch.all(delta[M:] == 7.0)
    y = O.linear(f64(A), f64(W), f64(bias))
    if epi < 2:
        assert rel_max(f64(out[:M]), O.gelu_tanh(y) if epi else y) <= 1e-2   # bf16 output
    else:
        want = f64(resid) + f64(gate) * y
        assert rel_max(f64(out[:M]), want) <= 1e-4
        if epi == 3:
            assert rel_max(f64(delta[:M]), want - f64(base)) <= 1e-2


# Stream-K shapes: the refine pass's one-candidate projections (1560 rows), a few tiles
# over a long K (13 pairs per tile), and two tiles over K = 9728 (about 38 pairs each).
SK_SHAPES = [(1560, 1536, 1536), (1560, 1536, 8960), (1560, 8960, 1536), (1560, 4608, 1536),
             (513, 512, 8960), (300, 256, 9728)]


@pytest.mark.parametrize("M,N,K", SK_SHAPES)
@pytest.mark.parametrize("epi", [0, 1, 2, 3])
def test_gemm_tc_stream_k_forced(model, M, N, K, epi):
    _gemm_case(model, M, N, K, epi, impl=4)


@pytest.mark.parametrize("M,N,K", SK_SHAPES[:2] + SK_SHAPES[-1:])
def test_gemm_stream_k_is_deterministic_and_matches_whole_tiles(model, M, N, K):
    """Cut tiles are summed in K order, so two runs agree bit for bit; whole-tile runs
    (impl 3) differ only by the fp32 summation order."""
    A = randn((M, K), 21)
    W = randn((N, K), 22, scale=K ** -0.5)
    resid = randn((M, N), 23, dtype=torch.float32)
    outs = []
    for impl in (4, 4, 3):
        out = torch.empty((M, N), dtype=torch.float32, device="cuda")
        fb.fb_op_gemm(model.handle, M, N, K, A, W, None, 2, out, resid, None, None, None, impl)
        outs.append(out)
    torch.cuda.synchronize()
    assert torch.equal(outs[0], outs[1])
    assert rel_max(f64(outs[0]), f64(outs[2])) <= 1e-5


@pytest.mark.parametrize("M,N,K,impl,blocks", [
    (1, 1536, 8960, 4, 12),      # 11.05 K blocks per pair, 13 contributors, one token
    (33, 1536, 8960, 0, 12),     # chunks that only some contributors finish
    (257, 1536, 8960, 4, 24),    # a second row of tiles with one token
    (640, 1536, 8960, 0, 34),    # ranges of two segments
    (2304, 1536, 8960, 4, 100),  # 54 tiles: up to three contributors
    (1040, 5120, 5120, 4, 80),   # ranges of three segments: one finisher
    (16, 1536, 8960, 3, 18),     # whole tiles of 16 tokens, eight parts
    (1560, 1536, 8960, 3, 47),   # three parts of 47, 47 and 46 K blocks
    (1040, 5120, 5120, 3, 40),   # two rounds: two parts in a ring of three accumulators
    (1400, 5120, 5120, 3, 40),   # two rounds: two parts in a ring of two
])
@pytest.mark.parametrize("epi", [0, 2])
def test_gemm_k_ranges(model, M, N, K, impl, blocks, epi):
    """Sums over K ranges joined in fp32, cut between SM pairs or kept in accumulators of
    their own: the error is that of the longest range. A 64-wide K block is four MMAs, each
    of which may truncate the running sum by one fp32 unit (1.2e-7 of it at most)."""
    A = randn((M, K), 71)
    W = randn((N, K), 72, scale=K ** -0.5)
    out = torch.empty((M, N), dtype=torch.float32 if epi else torch.bfloat16, device="cuda")
    for _ in range(2):  # (the second call finds the counters as the first left them)
        out.fill_(float("nan"))
        fb.fb_op_gemm(model.handle, M, N, K, A, W, None, epi, out, None, None, None, None, impl)
    torch.cuda.synchronize()
    want = A.double() @ W.double().T
    err = ((out.double() - want).norm() / want.norm()).item()
    # bf16 results: half a unit of 2^-8 at most
    assert err <= (1.2e-7 * blocks if epi else 2.0 ** -9)


@pytest.mark.parametrize("M,N,K", [
    (1, 1536, 8960),      # 13 contributors a tile, one token: most shares are empty
    (256, 1536, 8960),    # 13 contributors, full tiles
    (200, 512, 9728),     # two tiles, 38 contributors each
    (640, 1536, 8960),    # ranges that meet two cut tiles
    (1560, 1536, 8960),   # 42 tiles, two to four contributors
])
@pytest.mark.parametrize("epi", [0, 1, 2, 3])
def test_gemm_stream_k_handover(M, N, K, epi):
    """Contributors that hand their shares over to a tile's last one (as they do when one of
    them does not start): the sums keep their K order, so the result is that of the shared
    finish bit for bit, and the counters are zero again for the next launch."""
    A, W = randn((M, K), 61), randn((N, K), 62, scale=K ** -0.5)
    bias, gate = randn((N,), 63, dtype=torch.float32), randn((N,), 64, dtype=torch.float32)
    resid = randn((M, N), 65, dtype=torch.float32) if epi >= 2 else None
    outs = []
    with fb.Model(synth.TINY, synth.make_weights(synth.TINY)) as m:
        for handover in (False, True, False):
            out = torch.full((M, N), float("nan"), device="cuda",
                             dtype=torch.float32 if epi >= 2 else torch.bfloat16)
            delta = torch.full((M, N), float("nan"), dtype=torch.bfloat16, device="cuda")
            if handover:
                fb.fb_test_request_handover(m.handle, True)
            fb.fb_op_gemm(m.handle, M, N, K, A, W, bias, epi, out, resid,
                          gate if epi >= 2 else None, resid if epi == 3 else None,
                          delta if epi == 3 else None, 4)
            outs.append((out, delta))
        fb.fb_test_request_handover(m.handle, False)
    torch.cuda.synchronize()
    want = f64(A) @ f64(W).T + f64(bias)
    got = f64(outs[0][0])
    want = O.gelu_tanh(want) if epi == 1 else want if epi == 0 else f64(resid) + f64(gate) * want
    assert rel_max(got, want) <= (1e-2 if epi < 2 else 1e-4)
    for out, delta in outs[1:]:
        assert torch.equal(out, outs[0][0])
        if epi == 3:
            assert torch.equal(delta, outs[0][1])


def test_gemm_stream_k_on_several_streams():
    """Models on streams of their own, each launch sized for the whole device: two tiles with 38
    contributors each, so launches that run together can each hold part of a tile's pairs. Every
    call ends (well inside the wait limit) with the result of a call alone, bit for bit."""
    M, N, K, n = 200, 512, 9728, 4
    A, W = randn((M, K), 67), randn((N, K), 68, scale=K ** -0.5)
    models = [fb.Model(synth.TINY, synth.make_weights(synth.TINY)) for _ in range(n)]
    outs = [torch.zeros((M, N), dtype=torch.bfloat16, device="cuda") for _ in range(n + 1)]
    call = lambda m, out: fb.fb_op_gemm(m.handle, M, N, K, A, W, None, 0, out, None, None,  # noqa: E731
                                        None, None, 4)
    call(models[0], outs[n])
    torch.cuda.synchronize()
    errors = []

    def work(i):
        try:
            fb.fb_set_op_repeat(models[i].handle, 40)
            for _ in range(5):
                call(models[i], outs[i])
        except fb.FlashBonError as e:
            errors.append(str(e))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(n)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    for m in models:
        m.close()
    assert not errors
    for out in outs[:n]:
        assert torch.equal(out, outs[n])


@pytest.mark.parametrize("M,N,K,twin", [
    (1560, 1536, 8960, 4),   # 42 tiles, 140 K blocks: stream-K
    (640, 1536, 8960, 4),    # 18 tiles, 140 K blocks: stream-K
    (1560, 1536, 1536, 3),   # 24 K blocks: whole tiles
    (49920, 1536, 8960, 3),  # more tiles than SM pairs: whole tiles
    (8192, 1536, 8960, 3),   # 2.5 rounds but A and W (166 MB) larger than half of L2
    (2304, 1536, 8960, 3),   # one round, 40 idle K blocks a pair, but A and W are 68.8 MB
    (256, 5120, 13824, 4),   # 149 MB, but one row of tiles
])
def test_gemm_automatic_stream_k_choice(model, M, N, K, twin):
    """impl 0 takes the stream-K split where the last of at most four rounds of pair tiles
    leaves many K blocks idle and the operands are small or M is: its result is bit-identical
    to the forced variant it chose."""
    A = randn((M, K), 51)
    W = randn((N, K), 52, scale=K ** -0.5)
    resid = randn((M, N), 53, dtype=torch.float32)
    outs = []
    for impl in (0, twin):
        out = torch.empty((M, N), dtype=torch.float32, device="cuda")
        fb.fb_op_gemm(model.handle, M, N, K, A, W, None, 2, out, resid, None, None, None, impl)
        outs.append(out)
    torch.cuda.synchronize()
    assert torch.equal(outs[0], outs[1])


def test_gemm_stream_k_in_place_residual(model):
    M, N, K = 1560, 1536, 8960
    A, W = randn((M, K), 31), randn((N, K), 32, scale=K ** -0.5)
    h = randn((M, N), 33, dtype=torch.float32)
    h0 = f64(h)
    gate = randn((N,), 34, dtype=torch.float32)
    delta = torch.empty((M, N), dtype=torch.bfloat16, device="cuda")
    fb.fb_op_gemm(model.handle, M, N, K, A, W, None, 3, h, h, gate, h, delta, 4)
    torch.cuda.synchronize()
    want = h0 + f64(gate) * O.linear(f64(A), f64(W))
    assert rel_max(f64(h), want) <= 1e-4
    assert rel_max(f64(delta), want - h0) <= 1e-2


@pytest.mark.parametrize("M,N,K", [(300, 256, 128), (300, 384, 9728)])
def test_gemm_stream_k_forced_rejects(model, M, N, K):
    """Too few K blocks per SM pair, or N not a multiple of 256: an error, no launch."""
    A, W = randn((M, K), 41), randn((N, K), 42)
    out = torch.zeros((M, N), dtype=torch.bfloat16, device="cuda")
    with pytest.raises(fb.FlashBonError) as e:
        fb.fb_op_gemm(model.handle, M, N, K, A, W, None, 0, out, None, None, None, None, 4)
    assert e.value.status == fb.FB_ECUDA
    _gemm_case(model, M, N, K, 0, impl=0)   # the model is still usable


@pytest.mark.parametrize("budget", [3, 40])
def test_gemm_first_call_on_few_sms(budget):
    """The resident-cluster count is the device's, also when a process's first launch has a small
    or odd SM budget: on the whole device the stream-K split then still refuses a shape with
    fewer than four K blocks per SM pair (4 K blocks in all)."""
    code = f"""
import torch
from paper_2607_04461_gb300 import flashbon as fb, synth
m = fb.Model(synth.TINY, synth.make_weights(synth.TINY))
A, W = (torch.randn(n, 128).bfloat16().cuda() for n in (300, 256))
out = torch.empty(300, 256, dtype=torch.bfloat16, device="cuda")
run = lambda impl: fb.fb_op_gemm(m.handle, 300, 256, 128, A, W, None, 0, out, None, None, None, None, impl)
m.set_sm_budget({budget})
run(3)
m.set_sm_budget(0)
try:
    run(4)
    raise SystemExit("split taken")
except fb.FlashBonError as e:
    assert e.status == fb.FB_ECUDA
run(3)
torch.cuda.synchronize()
assert ((out.float() - A.float() @ W.float().T).abs().max() < 0.5).item()
"""
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr


@pytest.mark.parametrize("M,N,K", [(300, 256, 128), (77, 24, 40)])
@pytest.mark.parametrize("epi", [0, 1, 2, 3])
def test_gemm_simt(model, M, N, K, epi):
    _gemm_case(model, M, N, K, epi, impl=1)


def _gemm_case(model, M, N, K, epi, impl):
    A = randn((M, K), 1)
    W = randn((N, K), 2, scale=K ** -0.5)
    bias = randn((N,), 3, dtype=torch.float32)
    resid = randn((M, N), 4, dtype=torch.float32)
    gate = randn((N,), 5, dtype=torch.float32)
    base = randn((M, N), 6, dtype=torch.float32)
    out = torch.empty((M, N), dtype=torch.bfloat16 if epi < 2 else torch.float32, device="cuda")
    delta = torch.empty((M, N), dtype=torch.bfloat16, device="cuda")
    fb.fb_op_gemm(model.handle, M, N, K, A, W, bias, epi, out,
                  resid if epi >= 2 else None, gate if epi >= 2 else None,
                  base if epi == 3 else None, delta if epi == 3 else None, impl)
    torch.cuda.synchronize()
    y = O.linear(f64(A), f64(W), f64(bias))
    if epi == 0:
        assert rel_max(f64(out), y) <= 1e-2
    elif epi == 1:
        assert rel_max(f64(out), O.gelu_tanh(y)) <= 1e-2
    else:
        want = f64(resid) + f64(gate) * y
        assert rel_max(f64(out), want) <= 1e-4
        if epi == 3:
            assert rel_max(f64(delta), want - f64(base)) <= 1e-2


@pytest.mark.parametrize("M,N,K,impl", [
    (4999, 1536, 64, 0),     # the patch embedding: 2-SM kernel, one K block, ragged rows
    (3000, 128, 1536, 0),    # the padded head: 1-SM kernel, N = 128
    (300, 256, 128, 3),      # 2-SM whole tiles
    (1560, 1536, 8960, 4),   # 2-SM stream-K (cut tiles summed before the epilogue)
    (300, 256, 128, 2),      # 1-SM kernel forced
    (77, 24, 40, 1),         # CUDA-core kernel
])
@pytest.mark.parametrize("gated", [False, True])
def test_gemm_fp32_out_without_residual(model, M, N, K, impl, gated):
    """epi 2 with resid NULL: out = gate * (A W^T + bias) in fp32, every element written."""
    A = randn((M, K), 61)
    W = randn((N, K), 62, scale=K ** -0.5)
    bias = randn((N,), 63, dtype=torch.float32)
    gate = randn((N,), 64, dtype=torch.float32) if gated else None
    out = torch.full((M, N), float("nan"), dtype=torch.float32, device="cuda")
    fb.fb_op_gemm(model.handle, M, N, K, A, W, bias, 2, out, None, gate, None, None, impl)
    torch.cuda.synchronize()
    y = O.linear(f64(A), f64(W), f64(bias))
    want = f64(gate) * y if gated else y
    assert not torch.isnan(out).any()
    assert rel_max(f64(out), want) <= 1e-4


def test_gemm_in_place_residual(model):
    """out == resid and base == out (the block's last GEMM runs this way)."""
    M, N, K = 257, 256, 128
    A, W = randn((M, K), 11), randn((N, K), 12, scale=K ** -0.5)
    h = randn((M, N), 13, dtype=torch.float32)
    h0 = f64(h)
    hb = randn((M, N), 14, dtype=torch.float32)
    delta = torch.empty((M, N), dtype=torch.bfloat16, device="cuda")
    fb.fb_op_gemm(model.handle, M, N, K, A, W, None, 3, h, hb, None, h, delta)
    torch.cuda.synchronize()
    want = f64(hb) + O.linear(f64(A), f64(W))
    assert rel_max(f64(h), want) <= 1e-4
    assert rel_max(f64(delta), want - h0) <= 1e-2


ATTN_CASES = [
    # batch, Lq, Lkv, heads, dh, shared_kv
    (3, 150, 150, 2, 128, False),
    (2, 70, 40, 3, 64, True),
    (1, 1, 1, 1, 128, False),
    (2, 1560, 512, 2, 128, True),
    (1, 200, 333, 2, 64, False),
    (2, 1560, 1560, 2, 128, False),   # Wan2.1 self-attention length, ragged last tile
    (3, 256, 128, 1, 128, False),     # exact tile multiples
    (2, 129, 257, 2, 128, True),      # one row / one key past a tile
    # grids of more than one wave of 128-query CTAs take the persistent 256-query kernel
    # (P in TMEM)
    (4, 1560, 1560, 12, 128, False),
    (9, 600, 512, 12, 128, True),     # last CTA: tile A partly valid, tile B past Lq
    # the last key tile's MMAs cover only its 32-key chunks of real keys
    (2, 384, 192, 2, 128, False),     # 64 keys in the last tile; tile B starts at Lq
    (1, 300, 240, 2, 128, True),      # 112 keys: four chunks, the last one partial
    (2, 100, 193, 2, 128, False),     # 65 keys: three chunks
    # persistent 256-query CTAs: several items per CTA, one- and two-tile items mixed
    (12, 1560, 1560, 12, 128, False),
    (8, 300, 240, 12, 128, True),
]


@pytest.mark.parametrize("impl", [0, 3, 4], ids=["auto", "tc_q256", "tc_q256_persistent"])
def test_attention_large_logits(model, impl):
    """Scores spanning many powers of two exercise the rescaling of O."""
    batch, L, heads, dh = 2, 400, 2, 128
    D = heads * dh
    q = randn((batch * L, D), 41, scale=4.0)
    k = randn((batch * L, D), 42, scale=4.0)
    v = randn((batch * L, D), 43)
    o = torch.empty((batch * L, D), dtype=torch.bfloat16, device="cuda")
    fb.fb_op_attention(model.handle, q, D, k, D, v, D, o, D, batch, L, L, L, heads, dh, impl)
    torch.cuda.synchronize()
    qn, kn, vn, on = f64(q), f64(k), f64(v), f64(o)
    for b in range(batch):
        sl = slice(b * L, (b + 1) * L)
        want = O.attention(qn[sl].reshape(L, heads, dh), kn[sl].reshape(L, heads, dh),
                           vn[sl].reshape(L, heads, dh)).reshape(L, D)
        assert rel_max(on[sl], want) <= 2e-2


@pytest.mark.parametrize("impl", [0, 1, 2, 3, 4],
                         ids=["auto", "mma_sync", "tc_q128", "tc_q256", "tc_q256_persistent"])
@pytest.mark.parametrize("batch,Lq,Lkv,heads,dh,shared", ATTN_CASES)
def test_attention(model, batch, Lq, Lkv, heads, dh, shared, impl):
    D = heads * dh
    if impl >= 2 and dh != 128:
        z = torch.zeros((batch * max(Lq, Lkv), D), dtype=torch.bfloat16, device="cuda")
        with pytest.raises(fb.FlashBonError) as e:
            fb.fb_op_attention(model.handle, z, D, z, D, z, D, z, D, batch, Lq, Lkv, 0, heads,
                               dh, impl)
        assert e.value.status == fb.FB_EINVAL
        return
    q = randn((batch * Lq, D), 21)
    kvb = 1 if shared else batch
    k = randn((kvb * Lkv, D), 22)
    v = randn((kvb * Lkv, D), 23)
    o = torch.empty((batch * Lq, D), dtype=torch.bfloat16, device="cuda")
    fb.fb_op_attention(model.handle, q, D, k, D, v, D, o, D, batch, Lq, Lkv,
                       0 if shared else Lkv, heads, dh, impl)
    torch.cuda.synchronize()
    qn, kn, vn, on = f64(q), f64(k), f64(v), f64(o)
    for b in range(batch):
        kb = 0 if shared else b
        want = O.attention(qn[b * Lq:(b + 1) * Lq].reshape(Lq, heads, dh),
                           kn[kb * Lkv:(kb + 1) * Lkv].reshape(Lkv, heads, dh),
                           vn[kb * Lkv:(kb + 1) * Lkv].reshape(Lkv, heads, dh))
        got = on[b * Lq:(b + 1) * Lq]
        assert rel_max(got, want.reshape(Lq, D)) <= 2e-2
        assert np.abs(got - want.reshape(Lq, D)).mean() <= 2e-3


@pytest.mark.parametrize("batch,Lq,Lkv,heads,shared", [
    (1, 1100, 2000, 40, False),   # single-tile items among the cut ones, 2.3 rounds of items
    (3, 900, 1300, 14, False),    # 1.1 rounds: every item cut, ragged keys
    (2, 1200, 1700, 19, True),    # shared K/V, 1.25 rounds
    (5, 4096, 512, 12, True),     # four key tiles: not cut
])
def test_attention_key_split(model, batch, Lq, Lkv, heads, shared):
    """Items whose key range is cut between CTAs (equal shares per SM): against the fp64
    oracle on sampled heads, and bit for bit the same on a second and third call (the parts
    are added in CTA order; the flags are back at zero)."""
    cut = fb.fb_test_attention_split(model.handle, batch, Lq, Lkv, heads)
    assert (cut > 0) == (Lkv > 512)
    D = heads * 128
    q = randn((batch * Lq, D), 81)
    k = randn(((1 if shared else batch) * Lkv, D), 82)
    v = randn(((1 if shared else batch) * Lkv, D), 83)
    outs = []
    for _ in range(3):
        o = torch.empty((batch * Lq, D), dtype=torch.bfloat16, device="cuda")
        fb.fb_op_attention(model.handle, q, D, k, D, v, D, o, D, batch, Lq, Lkv,
                           0 if shared else Lkv, heads, 128)
        outs.append(o)
    torch.cuda.synchronize()
    assert torch.equal(outs[0], outs[1]) and torch.equal(outs[0], outs[2])
    for b in range(batch):
        kb = 0 if shared else b
        for hd in sorted({0, heads // 2, heads - 1}):
            c = slice(hd * 128, (hd + 1) * 128)
            want = O.attention(f64(q[b * Lq:(b + 1) * Lq, c])[:, None],
                               f64(k[kb * Lkv:(kb + 1) * Lkv, c])[:, None],
                               f64(v[kb * Lkv:(kb + 1) * Lkv, c])[:, None]).reshape(Lq, 128)
            got = f64(outs[0][b * Lq:(b + 1) * Lq, c])
            assert rel_max(got, want) <= 2e-2
            assert np.abs(got - want).mean() <= 2e-3


@pytest.mark.parametrize("batch,Lq,heads", [
    (40, 300, 11),   # one pair and a single tile with 44 rows
    (20, 640, 12),   # two pairs and a full single tile
    (14, 1400, 9),   # five pairs and a single tile
])
def test_attention_single_tiles_in_place(model, batch, Lq, heads):
    """More than 60 MB of K / V: the single last query tiles are numbered with their heads. The
    first, a middle and the last batch element's heads against the fp64 oracle; every row of
    the others agrees with the one-item-per-CTA kernel (bf16 rounding of P and O)."""
    D = heads * 128
    q, k, v = (randn((batch * Lq, D), 110 + i) for i in range(3))
    o, one = (torch.full((batch * Lq, D), float("nan"), dtype=torch.bfloat16, device="cuda")
              for _ in range(2))
    assert 4 * batch * Lq * D > 60e6
    assert fb.fb_test_attention_split(model.handle, batch, Lq, Lq, heads) == 0
    for out, impl in ((o, 0), (one, 3)):
        fb.fb_op_attention(model.handle, q, D, k, D, v, D, out, D, batch, Lq, Lq, Lq, heads, 128,
                           impl)
    torch.cuda.synchronize()
    assert rel_max(f64(o), f64(one)) <= 2e-2
    for b in (0, batch // 2, batch - 1):
        for hd in (0, heads - 1):
            r, c = slice(b * Lq, (b + 1) * Lq), slice(hd * 128, (hd + 1) * 128)
            want = O.attention(*(f64(x[r, c])[:, None] for x in (q, k, v))).reshape(Lq, 128)
            assert rel_max(f64(o[r, c]), want) <= 2e-2


@pytest.mark.parametrize("batch,Lq,Lkv,heads,impl", [
    (3, 900, 1300, 14, 0),   # every item cut into two parts
    (1, 2500, 4100, 6, 4),   # about three parts an item
    (12, 300, 700, 12, 4),   # whole items, one or two query tiles
    (2, 300, 700, 2, 2),     # 128-query CTAs
    (2, 300, 700, 2, 3),     # 256-query CTAs, one item each
])
def test_attention_masked_keys(model, batch, Lq, Lkv, heads, impl):
    """Scores of minus infinity through bias channels of q and k: the later half of the keys
    for every row (whole parts of cut items), the first 300 keys (two tiles and a piece) for
    one row per warp, and every key for another. The oracle sees the unmasked keys only; a row
    without any has no value (NaN), and its neighbours in the warp keep theirs."""
    cut = fb.fb_test_attention_split(model.handle, batch, Lq, Lkv, heads, impl)
    assert (cut > 0) == (Lkv > 700)
    D, lead, end = heads * 128, 300, Lkv // 2
    q, k, v = (randn((batch * n, D), 100 + i) for i, n in enumerate((Lq, Lkv, Lkv)))
    q4, k4 = q.view(batch, Lq, heads, 128), k.view(batch, Lkv, heads, 128)
    row = torch.arange(Lq, device="cuda")
    late, none = row % 32 == 9, row % 32 == 5
    q4[..., :3] = 0
    k4[..., :3] = 0
    q4[..., 0] = 1.0                      # keys end .. : score -inf for every row
    k4[:, end:, :, 0] = -float("inf")
    q4[:, none, :, 1] = -float("inf")     # rows with no key left
    k4[..., 1] = 1.0
    q4[:, late, :, 2] = 2.0 ** 120        # 2^120 * -2^120 overflows to -inf
    k4[:, :lead, :, 2] = -(2.0 ** 120)
    o = torch.full((batch * Lq, D), 7.0, dtype=torch.bfloat16, device="cuda")
    fb.fb_op_attention(model.handle, q, D, k, D, v, D, o, D, batch, Lq, Lkv, Lkv, heads, 128,
                       impl)
    torch.cuda.synchronize()
    late, none = late.cpu().numpy(), none.cpu().numpy()
    for b in sorted({0, batch - 1}):
        for hd in sorted({0, heads - 1}):
            c = slice(hd * 128, (hd + 1) * 128)
            got = f64(o[b * Lq:(b + 1) * Lq, c])
            qn = f64(q[b * Lq:(b + 1) * Lq, c])
            kn, vn = (f64(x[b * Lkv:b * Lkv + end, c]) for x in (k, v))
            for x in (qn, kn):
                x[:, :3] = 0.0            # the bias channels add nothing to an unmasked score
            kn[:, 1] = 0.0
            assert np.isnan(got[none]).all()
            for rows, first in ((~late & ~none, 0), (late, lead)):
                want = O.attention(qn[rows][:, None], kn[first:][:, None],
                                   vn[first:][:, None]).reshape(-1, 128)
                assert np.isfinite(got[rows]).all()
                assert rel_max(got[rows], want) <= 2e-2
                assert np.abs(got[rows] - want).mean() <= 2e-3


def test_attention_strided_qkv(model):
    """Self-attention reading q, k, v from one packed [rows][3D] buffer."""
    batch, L, heads, dh = 2, 97, 2, 128
    D = heads * dh
    qkv = randn((batch * L, 3 * D), 31)
    o = torch.empty((batch * L, D), dtype=torch.bfloat16, device="cuda")
    base = qkv.data_ptr()
    fb.fb_op_attention(model.handle, base, 3 * D, base + 2 * D, 3 * D, base + 4 * D, 3 * D, o,
                       D, batch, L, L, L, heads, dh)
    torch.cuda.synchronize()
    x = f64(qkv)
    for b in range(batch):
        r = x[b * L:(b + 1) * L]
        want = O.attention(r[:, :D].reshape(L, heads, dh), r[:, D:2 * D].reshape(L, heads, dh),
                           r[:, 2 * D:].reshape(L, heads, dh)).reshape(L, D)
        assert rel_max(f64(o)[b * L:(b + 1) * L], want) <= 2e-2


@pytest.mark.parametrize("ldo_pad,o_off", [(8, 0), (0, 8), (16, 0)],
                         ids=["row_stride_16B", "base_16B", "row_stride_32B"])
def test_attention_persistent_output_alignment(model, ldo_pad, o_off):
    """The persistent kernel stores O rows in 32-byte pieces only where the rows are
    32-byte aligned; a row stride or base aligned to 16 bytes only takes the 16-byte
    stores. Columns outside the heads' output stay untouched."""
    batch, L, heads, dh = 2, 300, 2, 128
    D = heads * dh
    ldo = D + ldo_pad
    q = randn((batch * L, D), 91)
    k = randn((batch * L, D), 92)
    v = randn((batch * L, D), 93)
    buf = torch.full((batch * L * ldo + o_off + 64,), 7.0, dtype=torch.bfloat16, device="cuda")
    o_ptr = buf.data_ptr() + 2 * o_off
    fb.fb_op_attention(model.handle, q, D, k, D, v, D, o_ptr, ldo, batch, L, L, L, heads, dh, 4)
    torch.cuda.synchronize()
    rows = buf[o_off:o_off + batch * L * ldo].view(batch * L, ldo)
    got = f64(rows[:, :D])
    if ldo_pad:
        assert torch.all(rows[:, D:] == 7.0)
    qn, kn, vn = f64(q), f64(k), f64(v)
    for b in range(batch):
        sl = slice(b * L, (b + 1) * L)
        want = O.attention(qn[sl].reshape(L, heads, dh), kn[sl].reshape(L, heads, dh),
                           vn[sl].reshape(L, heads, dh)).reshape(L, D)
        assert rel_max(got[sl], want) <= 2e-2


def test_pipe_probes_report_plausible_rates(model):
    """The measurement probes run and report values inside what the hardware allows: the
    tensor pipe at most 4096 MACs per SM clock (and at least half of it with no gap, less
    with a long gap), a special-function rate above zero and at most 64 per SM clock, and
    a TMEM load that takes clocks."""
    full = fb.fb_probe_mma_gap(0)
    gapped = fb.fb_probe_mma_gap(512)
    assert 2048 <= full <= 4096 * 1.01
    assert 0 < gapped < full
    for op in range(4):
        assert 0 < fb.fb_probe_mufu(op) <= 128
    for busy in (False, True):
        assert 10 < fb.fb_probe_tmem_load(busy) < 100000
    for form in range(14):
        for loaders, gap in ((0, 0), (7, 0)):
            assert 500 < fb.fb_probe_mma_mix(form, loaders, gap) < 4200
    with pytest.raises(fb.FlashBonError):
        fb.fb_probe_mma_mix(14)
    with pytest.raises(fb.FlashBonError):
        fb.fb_probe_mufu(4)
