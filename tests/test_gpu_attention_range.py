"""Long-sequence attention where a row's scores keep growing along the keys (the
running reference has to move, several times, and O with it), fall, or span
the exponent range, with ragged key tiles; and scores of one value."""

import pytest
import torch

from paper_2607_27842_gb300 import featfix as ff

from .gpu_helpers import rel_l2
from .test_gpu_ops import f64, randn

pytestmark = pytest.mark.gpu


# (text, image) tokens: key tiles cut inside the first half, inside the second
# half and right between them
@pytest.mark.parametrize("nt,ni", [(0, 1024), (77, 900), (5, 704), (130, 1000)])
@pytest.mark.parametrize("d", [64, 72, 128])
@pytest.mark.parametrize("span", [0.0, 30.0, 400.0])
def test_growing_scores(cuda, nt, ni, d, span):
    H, n = 2, nt + ni
    u = torch.zeros(d)
    u[::3] = 1.0
    u *= d ** 0.25 / u.norm()
    pos = torch.linspace(-0.5, 0.5, n)[:, None]
    sign = torch.where(torch.arange(n) % 2 == 0, 1.0, -1.0)[:, None]     # every other query sees falling scores
    # (a head's k and v are the same for every query; q k^T / sqrt(d) spans about +- span / 2)
    q = (sign * u)[:, None].expand(n, H, d)
    k = (pos * span * u)[:, None].expand(n, H, d)
    v = randn((n, H, d), "f32", 5, dev="cpu")
    qkv = torch.stack([q, k, v], 1).reshape(n, 3 * H * d).to(torch.bfloat16).to(cuda)
    out = torch.zeros((n, H * d), dtype=torch.bfloat16, device=cuda)
    ff.featfix_op_attention("bf16", qkv, out, 1, nt, ni, H, d)
    torch.cuda.synchronize()
    x = torch.from_numpy(f64(qkv)).reshape(n, 3, H, d)
    s = torch.einsum("qhd,khd->hqk", x[:, 0], x[:, 1]) / d ** 0.5
    ref = torch.einsum("hqk,khd->qhd", torch.softmax(s, -1), x[:, 2]).reshape(n, H * d)
    # P and the output are rounded to bf16 (2^-9 each, 1.7e-3 in the norm)
    assert rel_l2(f64(out), ref.numpy()) < 5e-3


# Large values under growing scores: against the running reference P is at most 2^8
# a key on average over any 64 keys and |v| at most 4 * 2^104, so O before the
# division is below 4096 * 2^8 * 2^106 = 2^126, inside fp32.
@pytest.mark.parametrize("d", [64, 72, 128])
@pytest.mark.parametrize("span", [20.0, 30.0])
def test_growing_scores_large_values(cuda, d, span):
    H, n = 2, 4096
    u = torch.zeros(d)
    u[::3] = 1.0
    u *= d ** 0.25 / u.norm()
    pos = torch.linspace(-0.5, 0.5, n)[:, None]
    q = u[None, None].expand(n, H, d)
    k = (pos * span * u)[:, None].expand(n, H, d)
    v = randn((n, H, d), "f32", 5, dev="cpu").clamp(-4, 4) * 2.0 ** 104
    qkv = torch.stack([q, k, v], 1).reshape(n, 3 * H * d).to(torch.bfloat16).to(cuda)
    out = torch.zeros((n, H * d), dtype=torch.bfloat16, device=cuda)
    ff.featfix_op_attention("bf16", qkv, out, 1, 0, n, H, d)
    torch.cuda.synchronize()
    x = torch.from_numpy(f64(qkv)).reshape(n, 3, H, d)
    s = torch.einsum("hd,khd->hk", x[0, 0], x[:, 1]) / d ** 0.5     # the same for every query
    ref = torch.einsum("hk,khd->hd", torch.softmax(s, -1), x[:, 2]).reshape(1, H * d).expand(n, -1)
    assert torch.isfinite(out).all()
    assert rel_l2(f64(out), ref.numpy()) < 5e-3     # as above
