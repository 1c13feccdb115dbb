"""bf16 dense layers at the edges of the tile shapes and of the rules that pick
them (single CTAs or CTA pairs, 128- or 256-wide tiles, several groups of row
blocks), against float64."""

import pytest
import torch

import oracle
from paper_2607_27842_gb300 import featfix as ff

from .gpu_helpers import rel_l2
from .test_gpu_ops import f64, randn

# The kernel a layer takes, restated from the dispatch: "pair128", "pair256" (CTA
# pairs, tiles 128 or 256 columns wide), "single" (a tile per CTA: its own
# epilogue where there is a residual or a history increment), "singles" (several
# tiles per CTA).  Outputs and gates of these tests allow the staged epilogues
# (16-byte aligned rows, at least 32 rows per gate sample).
def kernel(M, N, K, hist, sms):
    def waves(tiles, slots):
        return -(-tiles // slots)
    rem, m256 = N % 256, -(-M // 256)
    wide = -(-M // 128) * (N // 256) + (-(-rem // 128) * m256 if rem else 0)
    w256, w128 = (waves(m256 * -(-N // bn), sms // 2) for bn in (256, 128))
    if M >= 256 and w256 <= waves(wide, sms):
        if w128 <= w256:
            return "pair128"
        if w256 > 1 or K >= (4096 if hist else 1024):
            return "pair256"
    return "single" if wide <= sms else "singles"


# M, N, K, rows per gate sample, kernel without and with a history increment
SHAPES = [(256, 32, 64, 256, "pair128", "pair128"),        # one tile, mostly empty
          (257, 136, 72, 40, "pair128", "pair128"),        # a second row block of one row, 8 remainder columns
          (255, 256, 64, 255, "single", "single"),         # one row short of a pair
          (511, 264, 8, 32, "pair128", "pair128"),         # one k-step of 8
          (1024, 4608, 256, 256, "single", "single"),      # one wave, short reduction
          (1024, 4608, 1024, 200, "pair256", "single"),    # one wave, longer reduction
          (512, 8200, 4096, 200, "pair256", "pair256"),    # one wave, 8 remainder columns, K of 4096
          (2300, 1800, 136, 500, "single", "single"),      # remainder columns in swapped tiles
          (1000, 1160, 64, 100, "pair128", "pair128"),     # warps and blocks whose rows lie in two samples
          (300, 1288, 72, 33, "pair128", "pair128"),
          (900, 904, 136, 900, "pair128", "pair128"),
          (4333, 2056, 72, 100, "singles", "singles"),     # two waves where pairs would need three
          (4352, 3464, 72, 4352, "pair256", "pair256")]    # 17 row blocks: two full groups of eight and one


# the result is stored in bf16 (2^-9 relative, 1.7e-3 in the norm), the
# increment is the difference of two stored values rounded again
@pytest.mark.gpu
@pytest.mark.parametrize("M,N,K,rpb", [c[:4] for c in SHAPES])
@pytest.mark.parametrize("epilogue", ["bias", "gelu", "gated", "gated_history"])
def test_gemm_tiles(cuda, M, N, K, rpb, epilogue):
    a, w, bias = randn((M, K), "bf16", 1), randn((N, K), "bf16", 2, 0.1), randn(N, "bf16", 3)
    buf = torch.full((M + 1, N), 5.0, dtype=torch.bfloat16, device=cuda)
    out, kw, hist = buf[:M], {}, None
    y = f64(a) @ f64(w).T + f64(bias)
    if epilogue == "gelu":
        kw = dict(act=1)
        y = oracle.model.gelu_tanh(y)
    if epilogue.startswith("gated"):
        gate = randn((-(-M // rpb), 2 * N), "f32", 7)
        resid = randn((M, N), "bf16", 8)
        kw = dict(gate=gate[:, N:], gate_stride=2 * N, rows_per_batch=rpb, resid=resid)
        y = f64(resid) + f64(gate)[torch.arange(M).numpy() // rpb, N:] * y
    if epilogue == "gated_history":
        base, hist = randn((M, N), "bf16", 9), torch.full((M + 1, N), 5.0, dtype=torch.bfloat16, device=cuda)
        kw.update(hist_base=base, hist_out=hist[:M])
    ff.featfix_op_gemm("bf16", a, w, out, bias=bias, **kw)
    torch.cuda.synchronize()
    assert rel_l2(f64(out), y) < 4e-3
    assert torch.all(buf[M] == 5.0)
    if hist is not None:
        assert rel_l2(f64(hist)[:M], f64(out) - f64(base)) < 4e-3
        assert torch.all(hist[M] == 5.0)


# one tile per CTA: normal and swapped tiles, blocks cut by M and N, warps and
# blocks whose rows lie in two samples (rows per sample not multiples of 32)
SINGLE = [(4096, 1152, 200, 256), (130, 392, 1152, 130), (96, 264, 64, 32), (250, 520, 72, 33), (200, 1288, 64, 50),
          (255, 136, 64, 45), (2300, 1800, 136, 500)]
# the same forms on CTA pairs
PAIRED = [(1000, 1160, 64, 100), (300, 1288, 72, 33), (900, 904, 136, 900)]


@pytest.mark.parametrize("sms", [148, 152])
def test_cases_select_their_kernel(sms):
    for M, N, K, _, plain, hist in SHAPES:
        assert (kernel(M, N, K, False, sms), kernel(M, N, K, True, sms)) == (plain, hist), (M, N, K)
    for M, N, K, _ in SINGLE:
        assert kernel(M, N, K, False, sms) == kernel(M, N, K, True, sms) == "single", (M, N, K)
    for M, N, K, _ in PAIRED:
        assert kernel(M, N, K, False, sms) == kernel(M, N, K, True, sms) == "pair128", (M, N, K)


# bias and gate 16-byte aligned or not
@pytest.mark.gpu
@pytest.mark.parametrize("M,N,K,rpb", SINGLE + PAIRED)
@pytest.mark.parametrize("epilogue", ["resid", "gelu_gated", "gated_history"])
@pytest.mark.parametrize("shift", [0, 1])
def test_gemm_single_tile(cuda, M, N, K, rpb, epilogue, shift):
    a, w = randn((M, K), "bf16", 1), randn((N, K), "bf16", 2, 0.1)
    bias = randn(N + 8, "bf16", 3)[shift:shift + N]
    resid = randn((M, N), "bf16", 8)
    buf = torch.full((M + 1, N), 5.0, dtype=torch.bfloat16, device=cuda)
    hist = torch.full((M + 1, N), 5.0, dtype=torch.bfloat16, device=cuda)
    out, y, kw = buf[:M], f64(a) @ f64(w).T + f64(bias), {}
    if epilogue != "resid":
        gate = randn((-(-M // rpb), 2 * N + shift), "f32", 7)[:, N:2 * N]
        kw = dict(gate=gate, gate_stride=2 * N + shift, rows_per_batch=rpb)
        y = (oracle.model.gelu_tanh(y) if epilogue == "gelu_gated" else y) * f64(gate)[torch.arange(M).numpy() // rpb]
    if epilogue == "gelu_gated":
        kw["act"] = 1
    if epilogue == "gated_history":
        base = randn((M, N), "bf16", 9)
        kw.update(hist_base=base, hist_out=hist[:M])
    ff.featfix_op_gemm("bf16", a, w, out, bias=bias, resid=resid, **kw)
    torch.cuda.synchronize()
    assert rel_l2(f64(out), f64(resid) + y) < 4e-3
    assert torch.all(buf[M] == 5.0) and torch.all(hist[M] == 5.0)
    if epilogue == "gated_history":
        assert rel_l2(f64(hist)[:M], f64(out) - f64(base)) < 4e-3


# one tile per CTA with a history increment and no residual (nothing to load
# before the accumulator is ready): as above
@pytest.mark.gpu
@pytest.mark.parametrize("M,N,K,rpb", [(2300, 1800, 136, 500), (250, 520, 72, 33), (130, 392, 1152, 130), (40, 48, 64, 32)])
@pytest.mark.parametrize("gated", [False, True])
def test_gemm_single_tile_history_only(cuda, M, N, K, rpb, gated):
    a, w, bias, base = randn((M, K), "bf16", 1), randn((N, K), "bf16", 2, 0.1), randn(N, "bf16", 3), randn((M, N), "bf16", 9)
    buf = torch.full((2, M + 1, N), 5.0, dtype=torch.bfloat16, device=cuda)
    y, kw = f64(a) @ f64(w).T + f64(bias), {}
    if gated:
        gate = randn((-(-M // rpb), N), "f32", 7)
        kw = dict(gate=gate, gate_stride=N, rows_per_batch=rpb)
        y = y * f64(gate)[torch.arange(M).numpy() // rpb]
    ff.featfix_op_gemm("bf16", a, w, buf[0, :M], bias=bias, hist_base=base, hist_out=buf[1, :M], **kw)
    torch.cuda.synchronize()
    assert rel_l2(f64(buf[0, :M]), y) < 4e-3
    assert rel_l2(f64(buf[1, :M]), f64(buf[0, :M]) - f64(base)) < 4e-3
    assert torch.all(buf[:, M] == 5.0)


# The same product in a normal and in a swapped tile: the gate's product is rounded
# before the residual is added in both, so the outputs are the same bits.  (Added in
# one rounding, about 6 of a million stored values differ: 40 draws of 32640.)
@pytest.mark.gpu
def test_gemm_single_tile_same_bits(cuda):
    M, K = 255, 640                                     # below 256 rows: single CTAs; 256 columns normal, 128 swapped
    for seed in range(40):
        a, w, bias = randn((M, K), "bf16", 5 * seed), randn((128, K), "bf16", 5 * seed + 1, 0.05), randn(128, "bf16", 3)
        gate, resid, outs = randn((1, 128), "f32", 5 * seed + 2), randn((M, 128), "bf16", 5 * seed + 3), []
        for n in (1, 2):
            r = resid.repeat(1, n)
            out, hist = torch.empty_like(r), torch.empty_like(r)
            ff.featfix_op_gemm("bf16", a, w.repeat(n, 1), out, bias=bias.repeat(n), gate=gate.repeat(1, n),
                               gate_stride=128 * n, rows_per_batch=M, resid=r, hist_base=r, hist_out=hist)
            torch.cuda.synchronize()
            outs.append((out[:, :128], hist[:, :128]))
        assert torch.equal(outs[0][0], outs[1][0]) and torch.equal(outs[0][1], outs[1][1])
