"""The fp32 CUDA-core kernels at the edges of their tiles and dispatch rules,
against float64."""

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
            (1024, 4608, 65), (2, 6912, 1152)]


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
