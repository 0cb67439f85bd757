"""The tensor-core kernels at the edges of their tiles, against the fp64 oracle (relative
Frobenius error <= 1e-2 with the elementwise bound of tests/fqgpu.py, the bf16 tolerance of every
forward test): token counts around the 128- and 256-token tiles, an odd number of 128-row tiles (a
CTA pair whose second half has no rows), tiles split over K; the batch sizes of each decode tile
width with K ranges shorter than the ring; a rebuilt weight read by the call right after."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2403_06082_gb300 as fq  # noqa: E402
from fqgpu import DEV, DeviceLayer, activations, assert_parity, oracle_layer, reference  # noqa: E402

pytestmark = pytest.mark.gpu
BF16 = torch.bfloat16


@pytest.mark.parametrize("M", [65, 127, 128, 129, 255, 256, 257, 520])
@pytest.mark.parametrize("wl_key,name", [("single256", "single"), ("vit_b16_mlp", "fc1"),
                                         ("vit_b16_mlp", "fc2")])
def test_prefill_tiles(wl_key, name, M):
    # n = 288 is 3 tiles of 128 rows, 848 is 7, 3392 is 27; the ViT phases split K
    L = oracle_layer(wl_key, name)
    X = activations(wl_key, name, M)
    gamma = M % 2 == 0
    assert_parity(DeviceLayer(L).forward(X, gamma), reference(L, X, gamma), 1e-2)


@pytest.mark.parametrize("M", [1, 15, 16, 17, 32, 33, 64])
@pytest.mark.parametrize("wl_key,name", [("single256", "single"), ("vit_b16_mlp", "fc2")])
def test_decode_tiles(wl_key, name, M):
    L = oracle_layer(wl_key, name)
    X = activations(wl_key, name, M)
    gamma = M % 2 == 0
    assert_parity(DeviceLayer(L).forward(X, gamma), reference(L, X, gamma), 1e-2)


@pytest.mark.parametrize("sms", [1, 2, 3, 40])
def test_prefill_budgets(sms):
    """One SM (no CTA pair), one pair, an odd budget, a budget that changes the K splits."""
    L = oracle_layer("vit_b16_mlp", "fc1")
    X = activations("vit_b16_mlp", "fc1", 200)
    D = DeviceLayer(L)
    x = torch.from_numpy(X).to(DEV, BF16)
    y = torch.full((200, L.d_out), float("nan"), dtype=BF16, device=DEV)
    nb = fq.fq_workspace_bytes(200, L.d_in, L.n_in, L.n_out, L.d_out)
    ws = torch.zeros(nb, dtype=torch.uint8, device=DEV)
    fq.fq_linear_forward_sms(x, 200, L.d_in, D.T_in, D.C, D.T_out_t, L.d_out, None, y, ws, nb, sms)
    assert fq.fq_check(ws) == 0
    assert_parity(y.double().cpu().numpy(), reference(L, X), 1e-2)


@pytest.mark.parametrize("M", [100, 300])
def test_dense_reads_the_weight_just_rebuilt(M):
    """fq_dense_forward enqueued right after fq_reconstruct_weight reads the finished weight: the
    buffer holds NaN before, the two calls follow each other on the stream without a wait."""
    L = oracle_layer("vit_b16_mlp", "fc1")
    X = activations("vit_b16_mlp", "fc1", M)
    D = DeviceLayer(L)
    x = torch.from_numpy(X).to(DEV, BF16)
    nb = fq.fq_reconstruct_workspace_bytes(L.d_in, L.n_in, L.n_out, L.d_out)
    nd = fq.fq_dense_workspace_bytes(M, L.d_in, L.d_out)
    ws, wd = (torch.zeros(n, dtype=torch.uint8, device=DEV) for n in (nb, nd))
    W = torch.full((L.d_out, L.d_in), float("nan"), dtype=BF16, device=DEV)
    y = torch.empty(M, L.d_out, dtype=BF16, device=DEV)
    torch.cuda.synchronize()
    fq.fq_reconstruct_weight(D.T_in, D.C, D.T_out_t, L.d_in, L.d_out, None, W, ws, nb)
    fq.fq_dense_forward(x, M, L.d_in, W, L.d_out, y, wd, nd)
    assert fq.fq_check(ws) == 0 and fq.fq_check(wd) == 0
    assert_parity(y.double().cpu().numpy(), reference(L, X), 1e-2)


@pytest.mark.parametrize("M", [1, 300, 3000])
def test_rounded_activations_at_both_kernel_forms(M):
    """The rounding kernel with a block per token and with a warp per token (n_in <= 2048 and many
    tokens): identity codes and the trivial frames make y = bf16(Delta zbar), so y / Delta must be
    integers, the largest 7 (N = 4), and each equal to the rounded input but at ties."""
    d = 256
    g = np.random.Generator(np.random.PCG64(M))
    x = torch.from_numpy(g.standard_normal((M, d))).to(DEV, BF16)
    eye = torch.eye(d, dtype=BF16, device=DEV)
    codes = torch.eye(d, dtype=torch.uint8, device=DEV)
    one = torch.ones(d, dtype=torch.float16, device=DEV)
    words = torch.zeros(fq.fq_packed_words(d, d), dtype=torch.int32, device=DEV)
    C = fq.fq_pack(codes, one.view(torch.int16), (one * 0).view(torch.int16), d, d, words)
    mode = fq.FQ_BF16 | fq.FQ_ACT_BITS(4)
    nb = fq.fq_workspace_bytes(M, d, d, d, d, mode)
    ws = torch.zeros(nb, dtype=torch.uint8, device=DEV)
    y = torch.empty(M, d, dtype=BF16, device=DEV)
    fq.fq_linear_forward(x, M, d, eye, C, eye, d, None, y, ws, nb, mode)
    assert fq.fq_check(ws) == 0
    delta = x.double().abs().max() / 7
    q = x.double() / delta
    got = torch.round(y.double() / delta)
    off = got != torch.round(q)
    assert ((q - torch.floor(q) - 0.5).abs()[off] < 1e-5).all()
    assert got.abs().max() == 7


@pytest.mark.parametrize("M", [90, 150, 300])
def test_prefill_k_splits_repeat(M):
    """fc2 (848 and 3392 coefficients, K up to 53 blocks) at batches whose phases split K: calls on
    one workspace repeat bitwise (the splits' counters are left at zero) and match the oracle."""
    L = oracle_layer("vit_b16_mlp", "fc2")
    X = activations("vit_b16_mlp", "fc2", M)
    D = DeviceLayer(L)
    nb = fq.fq_workspace_bytes(M, L.d_in, L.n_in, L.n_out, L.d_out)
    ws = torch.zeros(nb, dtype=torch.uint8, device=DEV)
    first = D.forward(X, ws=ws)
    assert_parity(first, reference(L, X), 1e-2)
    for _ in range(3):
        np.testing.assert_array_equal(D.forward(X, ws=ws), first)
