"""Prefill under a budget of SMs that CTA pairs do not fill: one SM, and three, where the kernel
without pairs runs tiles of 128 or 256 tokens; against the fp64 oracle at the bf16 tolerance of every
forward test, around the tile widths, with and without rounded activations."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2403_06082_gb300 as fq  # noqa: E402
from fqgpu import DEV, DeviceLayer, activations, assert_parity, oracle_layer, reference  # noqa: E402

pytestmark = pytest.mark.gpu
BF16 = torch.bfloat16


def _forward(D, X, sms, mode=fq.FQ_BF16):
    L, M = D.L, X.shape[0]
    x = torch.from_numpy(X).to(DEV, BF16)
    y = torch.full((M, L.d_out), float("nan"), dtype=BF16, device=DEV)
    nb = fq.fq_workspace_bytes(M, L.d_in, L.n_in, L.n_out, L.d_out, mode)
    ws = torch.zeros(nb, dtype=torch.uint8, device=DEV)
    fq.fq_linear_forward_sms(x, M, L.d_in, D.T_in, D.C, D.T_out_t, L.d_out, None, y, ws, nb, sms,
                             mode)
    assert fq.fq_check(ws) == 0
    return y.double().cpu().numpy()


@pytest.mark.parametrize("sms", [1, 3])
@pytest.mark.parametrize("M", [128, 129, 255, 256, 257, 520])
@pytest.mark.parametrize("wl_key,name", [("single256", "single"), ("vit_b16_mlp", "fc2")])
def test_tile_widths_without_pairs(wl_key, name, M, sms):
    L = oracle_layer(wl_key, name)
    X = activations(wl_key, name, M)
    assert_parity(_forward(DeviceLayer(L), X, sms), reference(L, X), 1e-2)


@pytest.mark.parametrize("M", [16, 129, 300])
def test_rounded_activations_agree_over_budgets(M):
    """The code product is exact on rounded activations and both its kernels round u alike, so all
    budgets differ only by the analysis' and the synthesis' summation order."""
    L = oracle_layer("vit_b16_mlp", "fc1")
    D = DeviceLayer(L)
    X = activations("vit_b16_mlp", "fc1", M)
    mode = fq.FQ_BF16 | fq.FQ_ACT_BITS(8)
    full = _forward(D, X, 0, mode)
    for sms in (1, 3):
        assert_parity(_forward(D, X, sms, mode), full, 1e-2)
