"""The fp32 CUDA-core kernels and the row-wise LayerNorm at the edges of their tiles and dispatch rules,
against float64."""

import threading

import pytest
import torch

import oracle
from paper_2607_27842_gb300 import featfix as ff

from .gpu_helpers import rel_l2
from .test_gpu_ops import f64, randn

pytestmark = pytest.mark.gpu

# An fp32 dot product of K terms in s interleaved partial sums is off by at
# most about (K / s) u of the sum of the terms' magnitudes, in practice its
# square root: below 1e-6 of the result's norm for K <= 1200, s >= 2.
TOL = 1e-6


# the 16, 32, 64 and 128 tiles, K ranges split over 1, 2, 4 and 8 CTAs,
# remainders in every dimension, K not a multiple of four (4-byte copies), one
# row
F32_GEMM = [(1, 32, 64), (16, 32, 300), (17, 36, 68), (64, 128, 512), (64, 128, 1100), (31, 4, 258), (10, 512, 128),
            (65, 4100, 96), (130, 700, 70), (512, 1152, 200), (500, 3460, 36), (2000, 1540, 33), (1024, 4608, 68),
            (1024, 4608, 65), (2, 6912, 1152), (1175, 1156, 516), (1175, 1156, 517)]


@pytest.mark.parametrize("M,N,K", F32_GEMM)
@pytest.mark.parametrize("fused", [False, True])
def test_f32_gemm(cuda, M, N, K, fused):
    a, w, bias = randn((M, K), "f32", 1), randn((N, K), "f32", 2, 0.05), randn(N, "f32", 3)
    out = torch.full((M + 1, N), 7.0, device=cuda)
    if not fused:
        ff.featfix_op_gemm("f32", a, w, out[:M], bias=bias)
        ref = f64(a) @ f64(w).T + f64(bias)
    else:
        rpb = max(1, M // 3)
        gate = randn(((M + rpb - 1) // rpb, 2 * N), "f32", 7)
        resid, hist = randn((M, N), "f32", 8), torch.empty((M, N), device=cuda)
        ff.featfix_op_gemm("f32", a, w, out[:M], bias=bias, act=1, gate=gate[:, N:], gate_stride=2 * N,
                           rows_per_batch=rpb, resid=resid, hist_base=resid, hist_out=hist)
        y = oracle.model.gelu_tanh(f64(a) @ f64(w).T + f64(bias))
        ref = f64(resid) + f64(gate)[torch.arange(M).numpy() // rpb, N:] * y
        torch.cuda.synchronize()
        assert rel_l2(f64(hist), f64(out)[:M] - f64(resid)) < 1e-6
    torch.cuda.synchronize()
    assert rel_l2(f64(out)[:M], ref) < TOL
    assert torch.all(out[M] == 7.0)


# one and several tiles of 32 queries / 64 keys with remainders, text + image
# rows, every width class of the output columns; row strides that are not
# 16-byte multiples (scalar copies); bf16 head widths without a tensor-core
# kernel.  An output is a convex combination of values off by a few u (fp32:
# the exponents' error, |s| u, dominates) or by the storage rounding (bf16).
F32_ATTN = [("f32", 1, 0, 64, 4, 32, 0), ("f32", 2, 7, 90, 2, 72, 8), ("f32", 1, 0, 1, 3, 8, 0),
            ("f32", 2, 0, 256, 3, 72, 0), ("f32", 1, 33, 160, 2, 128, 4), ("f32", 3, 65, 1, 2, 64, 0),
            ("f32", 1, 5, 130, 2, 40, 3), ("f32", 1, 0, 97, 1, 104, 1), ("bf16", 2, 5, 100, 2, 96, 0),
            ("bf16", 1, 0, 70, 3, 40, 5), ("bf16", 1, 9, 200, 2, 8, 8)]


@pytest.mark.parametrize("dtype,B,nt,ni,H,d,pad", F32_ATTN)
def test_f32_attention(cuda, dtype, B, nt, ni, H, d, pad):
    C, n = H * d, nt + ni
    buf = randn((B * n, 3 * C + pad), dtype, 13)
    out = torch.full((B * n + 1, C), 3.0, dtype=buf.dtype, device=cuda)
    ff.featfix_op_attention(dtype, buf, out[:-1], B, nt, ni, H, d)
    torch.cuda.synchronize()
    rows = torch.tensor([[b * nt + t if t < nt else B * nt + b * ni + t - nt for t in range(n)] for b in range(B)])
    x = torch.from_numpy(f64(buf))[rows]
    q, k, v = (x[..., i * C:(i + 1) * C].reshape(B, n, H, d).transpose(1, 2) for i in range(3))
    ref = (torch.softmax(q @ k.transpose(2, 3) / d ** 0.5, -1) @ v).transpose(1, 2).reshape(B, n, C)
    assert rel_l2(f64(out)[rows], ref.numpy()) < (2e-6 if dtype == "f32" else 4e-3)
    assert torch.all(out[-1] == 3.0)


# ring depths and blocks per SM of every width class, samples that change inside
# a block, a last block and warp with few rows, one row; the last row counts of a
# row per warp on 152 SMs and the next ones; fp32 past the L2; unused row kept
LN = [("bf16", 1, 3072, 1), ("bf16", 4900, 128, 700), ("bf16", 6001, 1152, 250), ("bf16", 5003, 2048, 5003),
      ("bf16", 5000, 3072, 33), ("bf16", 77, 4096, 20), ("f32", 4999, 1536, 1000), ("f32", 5001, 2048, 7),
      ("bf16", 4864, 1536, 4864), ("bf16", 4865, 1536, 4865), ("bf16", 2433, 2048, 100), ("bf16", 1216, 4096, 1216),
      ("bf16", 1217, 4096, 1217), ("bf16", 5003, 4096, 5003), ("f32", 3648, 1024, 500), ("f32", 3649, 1024, 3649),
      ("f32", 2432, 2048, 2432), ("f32", 2435, 1536, 2435), ("f32", 12300, 2048, 12300)]


@pytest.mark.parametrize("dtype,rows,C,rpb", LN)
def test_ln_ring(cuda, dtype, rows, C, rpb):
    x = randn((rows, C), dtype, 1, 2.0) + 3.0
    mod = randn(((rows + rpb - 1) // rpb, 2 * C), "f32", 2, 0.1)
    out = torch.full((rows + 1, C), 9.0, dtype=x.dtype, device=cuda)
    ff.featfix_op_ln_modulate(dtype, x, out[:rows], rows, C, mod[:, :C], mod[:, C:], 2 * C, rpb)
    torch.cuda.synchronize()
    b = torch.arange(rows).numpy() // rpb
    ref = oracle.model.layer_norm(f64(x)) * (1 + f64(mod)[b, C:]) + f64(mod)[b, :C]
    assert rel_l2(f64(out)[:rows], ref) < (2e-6 if dtype == "f32" else 4e-3)
    assert torch.all(out[rows] == 9.0)


# Two threads, each with its own stream and row width, on one kernel instance:
# no call's launch may depend on the other's.  (The calls go through the C entry
# point with prepared arguments, so that they overlap.)
def test_ln_threads(cuda):
    rows, outs, calls, failed = 5000, [], [], [0, 0]
    for i, C in enumerate((1288, 1384)):
        x, mod = randn((rows, C), "bf16", 1, 2.0), randn((1, 2 * C), "f32", 2, 0.1)
        out, stream = torch.zeros_like(x), torch.cuda.Stream()
        ref = oracle.model.layer_norm(f64(x)) * (1 + f64(mod)[0, C:]) + f64(mod)[0, :C]
        outs.append((out, ref, x, mod, stream))
        calls.append((ff.DTYPE["bf16"], x.data_ptr(), out.data_ptr(), rows, C, mod.data_ptr(), mod.data_ptr() + 4 * C,
                      2 * C, rows, stream.cuda_stream))
    torch.cuda.synchronize()

    def work(i):
        op = ff.lib().featfix_op_ln_modulate
        for _ in range(6000):
            failed[i] += op(*calls[i]) != 0

    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert failed == [0, 0]
    for out, ref, *_ in outs:
        assert rel_l2(f64(out), ref) < 4e-3
