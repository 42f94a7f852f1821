"""Causal attention in each unit order and pairing of query tiles (attention_tc.cu): tile counts
odd and even, more units than SMs and fewer, last tiles with and without rowless warps."""
import pytest
import torch

from paper_2309_00754_gb300 import hydra as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nseq,P,heads", [
    (20, 300, 4),   # 3 tiles, 160 units: the first tile alone, a last tile of 44 rows
    (16, 390, 10),  # 4 tiles, a last tile of 6 rows
    (13, 640, 5),   # 5 tiles, 195 units: the first tile alone, whole tiles
    (3, 640, 4),    # 5 tiles, 36 units: the last tile alone
    (8, 900, 12),   # 8 tiles, 384 units of four lengths
    (40, 129, 5),   # 2 tiles, a last tile of one row
    (160, 97, 1),   # one tile, rows 96 .. in its last warp
    (5, 384, 16),   # 3 tiles, 160 units in rotated order, whole tiles
    (1, 300, 1),    # two units, the last tile alone and ragged
])
def test_causal_attention_orders(nseq, P, heads):
    g = torch.Generator(device="cuda").manual_seed(nseq * P)
    d = 128 * heads
    qkv = (1.28 * torch.randn(nseq * P, 3 * d, device="cuda", generator=g)).to(torch.bfloat16)
    out = torch.full((nseq * P, d), float("nan"), dtype=torch.bfloat16, device="cuda")
    H.hydra_causal_attention(qkv, nseq, P, heads, 128, out)
    q, k, v = qkv.double().view(nseq, P, 3, heads, 128).permute(2, 0, 3, 1, 4)
    z = q @ k.transpose(-1, -2) / 128 ** 0.5
    z.masked_fill_(torch.ones(P, P, dtype=torch.bool, device="cuda").triu(1), float("-inf"))
    ref = (torch.softmax(z, -1) @ v).transpose(1, 2).reshape(nseq * P, d)
    # bf16 probabilities (relative 2^-9 each) and a bf16 result: 2e-2 of max(1, |ref|), as
    # tests/test_gpu_llama.py states for this kernel
    err = ((out.double() - ref).abs() / ref.abs().clamp(min=1.0)).max().item()
    assert err <= 2e-2 and H.device_error(clear=True) == 0, err
