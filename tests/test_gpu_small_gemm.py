"""The linear of few token rows per stream (lora_gemm_small.cu) at the edges of its segments,
tiles, K items and K slices, against the oracle; and its order of summation, the tile kernel's
where K is one slice: the shared, stacked and three-stream forms, the fused epilogues and the
separate ones agree bit for bit, whichever kernel each takes."""
import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

from tests.helpers import TOL_LINEAR, TOL_LOGP, O, assert_abs, assert_rel, dev_bf16, dev_f32, dev_i32, f64, host_f64, synth
from paper_2309_00754_gb300 import build as B
from paper_2309_00754_gb300 import hydra as H

pytestmark = pytest.mark.gpu


def _problem(M, K, N, r, seed):
    g = lambda i, shape, std: synth.normal_bf16(1000 * seed + i, shape, std)  # noqa: E731
    x = [g(i, (M, K), 1.0) for i in range(3)]
    ab = [(g(10 + i, (r, K), 0.02), g(20 + i, (N, r), 0.02)) for i in range(2)] if r else [(None, None)] * 2
    return x, g(3, (N, K), 0.02), ab


def _dev(t):
    return None if t is None else dev_bf16(t)


@pytest.mark.parametrize("M,K,N,r,f32", [
    (1, 8, 8, 0, False),          # one row, one column chunk, one partial k-block
    (5, 136, 264, 8, True),       # an empty second segment; N and K tails
    (64, 1024, 520, 16, False),   # the longest K in one slice
    (64, 2048, 520, 16, False),   # two K slices of eight items each
    (65, 2184, 1032, 136, True),  # two LoRA items, the second of one k-block
    (128, 2048, 4104, 72, False),  # the largest single segment, a tail tile of one chunk
    (129, 1032, 4104, 72, True),  # two segments per stream, 34 256-column tiles
    (257, 5128, 1288, 8, False),  # two slices again: 18 tiles
    (257, 520, 1288, 8, False),   # three segments per stream: a pair of the off and the on stream
    (384, 264, 12288, 16, False),  # more tiles than the chip holds at once
    (448, 200, 520, 8, True),
    (512, 136, 5120, 8, False),  # the most rows: full segments, four per stream
    (100, 4096, 12288, 16, False),  # two streams take this kernel, three the tile kernel
    (300, 512, 12288, 136, True),  # the same, two LoRA items
    (224, 640, 10240, 200, False),  # one input: the drain's buffers beside the LoRA items
    (40, 1024, 22016, 32, False),  # one stream takes the tile kernel
])
def test_few_rows_against_oracle_and_one_order_of_sums(M, K, N, r, f32):
    x, W, ab = _problem(M, K, N, r, seed=M + K)
    dt = torch.float32 if f32 else torch.bfloat16
    d, dW = [dev_bf16(t) for t in x], dev_bf16(W)
    dab = [(_dev(a), _dev(b)) for a, b in ab]
    new = lambda: torch.full((M, N), float("nan"), dtype=dt, device="cuda")  # noqa: E731
    ws = torch.empty(max(1, H.lora_linear_tri_workspace_size(M, r)), dtype=torch.uint8, device="cuda")

    def two(xa, xb, a, b, want=(True, True)):
        y = [new() if w else None for w in want]
        H.hydra_lora_linear(xa, xb, dW, a, b, 2.0, y[0], y[1], ws, algo=1)
        return y

    tri = [new() for _ in range(3)]
    H.hydra_lora_linear_tri(d[0], d[1], d[2], dW, *dab[0], *dab[1], 2.0, *tri, ws)
    st = two(d[0], d[1], *dab[0])
    sh = two(d[1], None, *dab[0])
    crit = two(d[2], None, *dab[1], want=(False, True))
    off = two(d[0], None, *dab[0], want=(True, False))
    assert torch.equal(st[1], sh[1]) and torch.equal(off[0], st[0])
    assert torch.equal(tri[0], st[0]) and torch.equal(tri[1], st[1]) and torch.equal(tri[2], crit[1])
    # against fp64, fp32 sums of bf16 products in another order: 1e-4 as for the tile kernel's fp32
    # outputs. u is the library's own (hydra_lora_down, tested by itself): where it rounds to bf16
    # the other way than the oracle's, y moves by ulp(u) |B|, up to 2^-6 * 0.1 = 1.6e-3
    tol = 1e-4 if f32 else TOL_LINEAR
    for y, i, (a, b) in ((tri[0], 0, (None, None)), (tri[1], 1, dab[0]), (tri[2], 2, dab[1])):
        ref = f64(x[i]) @ f64(W).T
        if a is not None:
            u = torch.empty(M, r, dtype=torch.bfloat16, device="cuda")
            H.hydra_lora_down(d[i], a, 2.0, u)
            ref += host_f64(u) @ host_f64(b).T
        assert_rel(host_f64(y), ref if f32 else O.round_bf16(ref), tol, f"stream {i}")


@pytest.mark.parametrize("M,N,shared", [(33, 512, False), (97, 512, True), (128, 768, False), (200, 392, False),
                                        (300, 392, True), (97, 22016, False), (7, 22016, True)])
def test_few_rows_fused_epilogues(M, N, shared):
    """SwiGLU, rotary (N past the rotated columns, a partial last head) and residual epilogues
    equal the plain linear followed by the separate kernel, bit for bit (two K slices; at 22016
    columns one, and 160-column tiles of five boxes)."""
    K, r, P = 2184, 16, 50
    x, W, ab = _problem(M, K, N, r, seed=7 * M + N)
    d, dW, dB = [dev_bf16(t) for t in x], dev_bf16(W), dev_bf16(ab[0][1])
    xo = None if shared else d[1]
    u = dev_bf16(synth.normal_bf16(99, (M, r), 2.0))
    lin = [torch.empty(M, N, dtype=torch.bfloat16, device="cuda") for _ in range(2)]
    H.hydra_dual_linear(d[0], xo, dW, u, dB, lin[0], lin[1], algo=1)
    h0 = synth.normal_f32(98, (2, M, N), 3.0)
    h, want = dev_f32(h0), dev_f32(h0)
    H.hydra_dual_linear_ex(d[0], xo, dW, u, dB, h[0], h[1], H.EPI_RESIDUAL)
    for i in range(2):
        H.hydra_residual_add(want[i].view(-1), lin[i].view(-1))
    assert torch.equal(h, want)
    d_rot = 128
    got = [torch.empty(M, N, dtype=torch.bfloat16, device="cuda") for _ in range(2)]
    table = torch.empty(P, 64, 2, device="cuda")
    H.hydra_rope_table(P, 128, 10000.0, table)
    H.hydra_dual_linear_rope(d[0], xo, dW, u, dB, got[0], got[1], P, 2 * d_rot, 128, table)
    if N % 256 == 0:  # W rows as interleaved gate / up blocks of 128
        m = [torch.empty(M, N // 2, dtype=torch.bfloat16, device="cuda") for _ in range(2)]
        H.hydra_dual_linear_ex(d[0], xo, dW, u, dB, m[0], m[1], H.EPI_SWIGLU)
        for i in range(2):
            gu = lin[i].view(M, N // 256, 2, 128).transpose(1, 2).reshape(M, N).contiguous()
            ref = torch.empty_like(m[i])
            H.hydra_swiglu(gu, ref)
            assert torch.equal(m[i], ref)
    for i in range(2):
        H.hydra_rope(lin[i], d_rot, 128, P, 10000.0)
        assert torch.equal(got[i], lin[i])
    assert H.device_error(clear=True) == 0


def test_fused_silu_has_the_operators_bits_for_every_bf16_gate():
    """W's first column is every bf16 value (infinities, NaN and both zeros among them) and x picks
    it out: the epilogue's branch-free quotient against hydra_swiglu's division operator."""
    F, K, M = 65536, 8, 3
    gate = torch.arange(F, device="cuda", dtype=torch.int32).to(torch.int16).view(torch.bfloat16)
    W = torch.zeros(F // 128, 2, 128, K, dtype=torch.bfloat16, device="cuda")
    W[:, 0, :, 0] = gate.view(-1, 128)
    W[:, 1, :, 0] = 1.0
    x = torch.zeros(M, K, dtype=torch.bfloat16, device="cuda")
    x[:, 0] = 1.0
    m = [torch.empty(M, F, dtype=torch.bfloat16, device="cuda") for _ in range(2)]
    H.hydra_dual_linear_ex(x, x, W.view(2 * F, K), None, None, m[0], m[1], H.EPI_SWIGLU)
    # the tensor core's sum 1 * g + 0 keeps every g but -0, which it makes +0
    g = torch.where(gate == 0, torch.zeros_like(gate), gate)
    ref = torch.empty(1, F, dtype=torch.bfloat16, device="cuda")
    H.hydra_swiglu(torch.cat([g, torch.ones_like(g)]).view(1, 2 * F), ref)
    for y in m:  # bits: a zero's sign counts
        assert bool(((y.view(torch.int16) == ref.view(torch.int16)) | (y.isnan() & ref.isnan())).all())
    assert int(ref.isnan().sum()) >= 254  # the NaN patterns, and -inf / inf


def test_silu_has_the_operators_bits_for_every_fp32_input(tmp_path):
    """The bf16 outputs above hide most last-bit differences of the quotient: here it is compared
    in fp32, over all 2^32 inputs."""
    here = os.path.dirname(os.path.abspath(__file__))
    so = str(tmp_path / "silu_bits.so")
    subprocess.run([B._nvcc(), *B.ARCH, *B.NVCC_FLAGS, "-I", B.CSRC, "-shared", os.path.join(here, "silu_bits.cu"), "-o", so],
                   check=True)
    differ = torch.zeros(1, dtype=torch.int64, device="cuda")
    rc = ctypes.CDLL(so).count_silu_bits(ctypes.c_void_p(differ.data_ptr()),
                                         ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == 0 and int(differ) == 0


@pytest.mark.parametrize("M,K,V", [(1, 8, 8), (32, 136, 1000), (33, 1032, 264), (64, 4096, 40000)])
def test_log_softmax_of_both_streams_in_one_tile(M, K, V):
    """Up to 64 rows of two streams without LoRA share 128-row tiles (also more tiles than SMs);
    the same rows in a call of 200 rows take CTA pairs, one stream a tile, with the same sums in
    the same order: equal bits."""
    g = lambda i, shape, std: dev_bf16(synth.normal_bf16(31 * M + i, shape, std))  # noqa: E731
    h, W = [g(i, (200, K), 1.0) for i in range(2)], g(2, (V, K), 0.05)
    ids = dev_i32(synth.randint(77 + M, (200,), 0, V))

    def run(m):
        ws = torch.empty(H.lm_head_logprobs_workspace_size(1, m, V, 0), dtype=torch.uint8, device="cuda")
        out = [torch.full((m,), float("nan"), device="cuda") for _ in range(5)]
        H.hydra_lm_head_logprobs(h[0][:m], h[1][:m], W, None, None, 1.0, ids[:m], None, None, 0.1, 1, m,
                                 out[0], out[1], out[2], ws, lse_actor=out[3], lse_ref=out[4])
        return out

    for got, want in zip(run(M), run(200)):
        assert torch.equal(got, want[:M])
    assert H.device_error(clear=True) == 0


@pytest.mark.parametrize("M,K,V,r", [(1, 136, 264, 8), (60, 520, 1000, 16), (100, 1032, 520, 0), (128, 136, 4104, 136)])
def test_log_softmax_of_a_row_segment_per_stream(M, K, V, r):
    """Log-softmax partials of a pair that holds both streams (65 to 128 rows, or LoRA): three
    warps per row merge their chunks; against the oracle, two streams, the last tile partial."""
    x, W, ab = _problem(M, K, V, r, seed=3 * M + V)
    A, B = ab[0]
    ids = synth.randint(78 + M, (M,), 0, V)
    ws = torch.empty(H.lm_head_logprobs_workspace_size(1, M, V, r), dtype=torch.uint8, device="cuda")
    out = [torch.full((M,), float("nan"), device="cuda") for _ in range(5)]
    H.hydra_lm_head_logprobs(dev_bf16(x[0]), dev_bf16(x[1]), dev_bf16(W), _dev(A), _dev(B), 2.0, dev_i32(ids), None,
                             None, 0.1, 1, M, out[0], out[1], out[2], ws, lse_actor=out[3], lse_ref=out[4])
    z_ref, z_act = O.dual_lora_linear(f64(x[0]), f64(x[1]), f64(W), None if A is None else f64(A),
                                      None if B is None else f64(B), 2.0, out_bf16=False)
    for got, z in ((out[0], z_act), (out[1], z_ref)):
        assert_abs(host_f64(got), O.log_softmax_gather(z, ids)[0], TOL_LOGP, "logp")
    assert H.device_error(clear=True) == 0


def test_a_row_has_the_same_bits_among_few_rows_and_among_many():
    """One K slice sums as the tile kernel does: the first rows of a call of 600, and of 97 alone."""
    K, N, r = 1032, 12296, 16
    x, W, ab = _problem(600, K, N, r, seed=9)
    d, dW = [dev_bf16(t) for t in x], dev_bf16(W)
    A, B = dev_bf16(ab[0][0]), dev_bf16(ab[0][1])
    u = torch.empty(600, r, dtype=torch.bfloat16, device="cuda")
    H.hydra_lora_down(d[1], A, 2.0, u)

    def run(m, shared):
        y = [torch.empty(m, N, device="cuda") for _ in range(2)]
        H.hydra_dual_linear(d[1][:m] if shared else d[0][:m], None if shared else d[1][:m], dW, u[:m], B, y[0], y[1], algo=1)
        return y

    for shared in (False, True):
        many = run(600, shared)
        for m in (20, 97, 128, 200, 300):
            for a, b in zip(run(m, shared), many):
                assert torch.equal(a, b[:m]), (m, shared)


def test_off_rows_ignore_a_non_finite_lora_factor():
    """A pair of an off and an on segment: infinities in B reach the LoRA-on rows alone."""
    M, K, N, r = 40, 256, 264, 16
    x, W, ab = _problem(M, K, N, r, seed=5)
    d, dW = [dev_bf16(t) for t in x], dev_bf16(W)
    A, B = dev_bf16(ab[0][0]), torch.full((N, r), float("inf"), dtype=torch.bfloat16, device="cuda")
    ws = torch.empty(H.lora_linear_workspace_size(M, r), dtype=torch.uint8, device="cuda")
    y = [torch.empty(M, N, device="cuda") for _ in range(2)]
    H.hydra_lora_linear(d[0], d[1], dW, A, B, 2.0, y[0], y[1], ws)
    assert np.all(np.isfinite(host_f64(y[0]))) and not bool(torch.isfinite(y[1]).any())


@pytest.mark.parametrize("M,K,N,r,shared", [(1, 4096, 4096, 16, False), (8, 520, 1048, 64, False), (16, 1032, 264, 8, True)])
def test_gemv_beside_its_lora_down_matches_the_two_calls_in_turn(M, K, N, r, shared):
    """hydra_lora_linear's GEMV starts before its lora_down has ended; hydra_lora_down followed by
    hydra_dual_linear runs the same arithmetic in turn: the same bits, also with new inputs in the
    same buffers, call after call."""
    x, W, ab = _problem(M, K, N, r, seed=17 + M)
    dW, A, B = dev_bf16(W), dev_bf16(ab[0][0]), dev_bf16(ab[0][1])
    buf = [torch.empty(M, K, dtype=torch.bfloat16, device="cuda") for _ in range(2)]
    ws = torch.empty(H.lora_linear_workspace_size(M, r), dtype=torch.uint8, device="cuda")
    got = [[torch.empty(M, N, dtype=torch.bfloat16, device="cuda") for _ in range(2)] for _ in range(40)]
    for i, y in enumerate(got):
        for j in range(2):
            buf[j].copy_(dev_bf16(x[(i + j) % 3]))
        H.hydra_lora_linear(buf[0], None if shared else buf[1], dW, A, B, 2.0, y[0], y[1], ws)
    for i in range(3):
        xs = [dev_bf16(x[(i + j) % 3]) for j in range(2)]
        xo = xs[0] if shared else xs[1]
        u = torch.empty(M, r, dtype=torch.bfloat16, device="cuda")
        H.hydra_lora_down(xo, A, 2.0, u)
        torch.cuda.synchronize()
        y = [torch.empty(M, N, dtype=torch.bfloat16, device="cuda") for _ in range(2)]
        H.hydra_dual_linear(xs[0], None if shared else xo, dW, u, B, y[0], y[1])
        for k in range(i, 40, 3):
            assert torch.equal(got[k][0], y[0]) and torch.equal(got[k][1], y[1])


@pytest.mark.parametrize("M,K,N,r,form", [
    (20, 2048, 776, 16, "two"),     # fewer than 64 rows: the lora_down that is not streamed; two K slices
    (40, 1024, 4096, 8, "shared"),  # one slice
    (40, 4096, 1032, 16, "three"),
    (64, 4096, 8192, 16, "two"),    # the streamed lora_down from here on
    (97, 4096, 1024, 64, "three"),  # two slices
    (97, 4096, 4096, 16, "shared"),
    (97, 2048, 12288, 16, "two"),   # one slice, more tiles than the chip holds at once
    (300, 2048, 520, 136, "two"),   # two slices, two LoRA items
    (300, 4096, 4096, 64, "shared"),
    (300, 1024, 1032, 8, "three"),
])
def test_few_rows_beside_its_lora_down_with_new_inputs_in_the_same_buffers(M, K, N, r, form):
    """The few-rows kernel reads x and W before the lora_down of its call has ended. x is written anew
    before each call by a kernel that lets its dependents start at once (RMSNorm), W every other call;
    call after call without a synchronisation equals the same calls one at a time."""
    n = {"shared": 1, "two": 2, "three": 3}[form]
    h = [[dev_f32(synth.normal_f32(500 + 3 * i + j, (M, K), 1.0)) for j in range(n)] for i in range(3)]
    W = [dev_bf16(synth.normal_bf16(520 + i, (N, K), 0.02)) for i in range(2)]
    A = [dev_bf16(synth.normal_bf16(530 + i, (r, K), 0.02)) for i in range(2)]
    Bm = [dev_bf16(synth.normal_bf16(540 + i, (N, r), 0.02)) for i in range(2)]
    one = torch.ones(K, dtype=torch.bfloat16, device="cuda")
    x = [torch.empty(M, K, dtype=torch.bfloat16, device="cuda") for _ in range(n)]
    w = torch.empty_like(W[0])
    ws = torch.empty(H.lora_linear_tri_workspace_size(M, r), dtype=torch.uint8, device="cuda")

    def call(i, y):
        if i % 2 == 0:
            w.copy_(W[i // 2 % 2])
        for j in range(n):
            H.hydra_rmsnorm(h[i % 3][j], one, 1e-6, x[j])
        if n == 3:
            H.hydra_lora_linear_tri(x[0], x[1], x[2], w, A[0], Bm[0], A[1], Bm[1], 2.0, *y, ws)
        else:
            H.hydra_lora_linear(x[0], x[1] if n == 2 else None, w, A[0], Bm[0], 2.0, y[0], y[1], ws, algo=1)

    new = lambda: [torch.full((M, N), float("nan"), dtype=torch.bfloat16, device="cuda") for _ in range(max(2, n))]  # noqa: E731
    want = []
    for i in range(12):  # every combination of x and W
        want.append(new())
        call(i, want[i])
        torch.cuda.synchronize()
    got = [new() for _ in range(36)]
    torch.cuda.synchronize()
    for i, y in enumerate(got):
        call(i, y)
    torch.cuda.synchronize()
    for i, y in enumerate(got):
        assert all(torch.equal(a, b) for a, b in zip(y, want[i % 12])), i
    if n < 3:  # and the two kernels in turn
        u = torch.empty(M, r, dtype=torch.bfloat16, device="cuda")
        y = new()
        H.hydra_lora_down(x[n - 1], A[0], 2.0, u)
        torch.cuda.synchronize()
        H.hydra_dual_linear(x[0], x[1] if n == 2 else None, w, u, Bm[0], y[0], y[1], algo=1)
        assert all(torch.equal(a, b) for a, b in zip(y, got[-1]))
    assert H.device_error(clear=True) == 0
