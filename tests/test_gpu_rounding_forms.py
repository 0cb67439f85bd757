"""The rounding of the activations with a warp or a block per token, on both sides of the sizes where
one takes over from the other.  Identity codes and trivial frames make y = bf16(Delta zbar), so y /
Delta rounds to zbar: the nearest integer to x / Delta, or its neighbour at a tie of the fp32 quotient
(within 2^-20 of a half: quotients stay below 8 and carry two fp32 roundings)."""
import pytest

torch = pytest.importorskip("torch")

import paper_2403_06082_gb300 as fq  # noqa: E402

pytestmark = pytest.mark.gpu
BF16 = torch.bfloat16


@pytest.mark.parametrize("d", [16, 512, 528, 2304, 2320])
@pytest.mark.parametrize("per_sm", [8, 32, 64])
@pytest.mark.parametrize("less", [0, 1])
def test_rounded_values(d, per_sm, less):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    M = per_sm * sms - less
    g = torch.Generator(device="cuda").manual_seed(d + M)
    x = torch.randn(M, d, generator=g, device="cuda").to(BF16)
    eye = torch.eye(d, dtype=BF16, device="cuda")
    one = torch.ones(d, dtype=torch.float16, device="cuda")
    words = torch.zeros(fq.fq_packed_words(d, d), dtype=torch.int32, device="cuda")
    C = fq.fq_pack(eye.to(torch.uint8), one.view(torch.int16), (one * 0).view(torch.int16), d, d,
                   words)
    mode = fq.FQ_BF16 | fq.FQ_ACT_BITS(4)
    nb = fq.fq_workspace_bytes(M, d, d, d, d, mode)
    ws = torch.zeros(nb, dtype=torch.uint8, device="cuda")
    y = torch.full((M, d), float("nan"), dtype=BF16, device="cuda")
    fq.fq_linear_forward(x, M, d, eye, C, eye, d, None, y, ws, nb, mode)
    assert fq.fq_check(ws) == 0
    delta = x.double().abs().max() / 7
    q = x.double() / delta
    got = torch.round(y.double() / delta)
    off = got != torch.round(q)
    assert ((q - torch.floor(q) - 0.5).abs()[off] <= 2.0 ** -20).all()
    assert got.abs().max() == 7
