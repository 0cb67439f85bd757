"""One zero-filled workspace over calls that differ in batch size, layer and path: what a call needs
from the one before lies in the header at fixed places, so every result is bitwise that of a fresh
workspace.  Batches and layers are those whose phases split K (their tiles are counted in the
workspace); outputs start as NaN, so a tile that is left unwritten shows."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2403_06082_gb300 as fq  # noqa: E402
from fqgpu import DEV, DeviceLayer, activations, assert_parity, oracle_layer, reference  # noqa: E402

pytestmark = pytest.mark.gpu
BF16 = torch.bfloat16
FC1, FC2, SMALL = ("vit_b16_mlp", "fc1"), ("vit_b16_mlp", "fc2"), ("single256", "single")


def _zeros(nbytes):
    return torch.zeros(nbytes, dtype=torch.uint8, device=DEV)


@pytest.mark.parametrize("calls", [
    [(FC2, 200), (FC2, 100), (FC2, 300), (FC2, 100)],          # the batch size changes
    [(FC2, 100), (FC1, 100), (SMALL, 100), (FC2, 129)],        # the layer changes
    [(FC2, 200), (FC2, 16), (FC2, 100), (FC1, 64), (FC1, 90)]  # fused calls between
], ids=["batch", "layer", "decode"])
def test_forward_calls_share_a_workspace(calls):
    layers = {k: (L, DeviceLayer(L)) for k in {k for k, _ in calls} for L in [oracle_layer(*k)]}
    ws = _zeros(max(fq.fq_workspace_bytes(M, L.d_in, L.n_in, L.n_out, L.d_out)
                    for k, M in calls for L, _ in [layers[k]]))
    for k, M in calls:
        L, D = layers[k]
        X = activations(*k, M)
        got = D.forward(X, ws=ws)
        assert_parity(got, reference(L, X), 1e-2)
        np.testing.assert_array_equal(got, D.forward(X))


def test_group_of_unlike_layers_above_the_fused_batch():
    M = 100
    Ls = [oracle_layer(*k) for k in (FC2, FC1, SMALL)]
    Ds = [DeviceLayer(L) for L in Ls]
    Xs = [activations(*k, M) for k in (FC2, FC1, SMALL)]
    ys = [torch.full((M, L.d_out), float("nan"), dtype=BF16, device=DEV) for L in Ls]
    group = [fq.Layer(torch.from_numpy(X).to(DEV, BF16), L.d_in, D.T_in, D.C, D.T_out_t, L.d_out,
                      None, y) for L, D, X, y in zip(Ls, Ds, Xs, ys)]
    ws = _zeros(fq.fq_group_workspace_bytes(M, group))
    for _ in range(2):
        for y in ys:
            y.fill_(float("nan"))
        fq.fq_linear_forward_group(M, group, ws, ws.numel())
        assert fq.fq_check(ws) == 0
        for D, X, y in zip(Ds, Xs, ys):
            np.testing.assert_array_equal(y.double().cpu().numpy(), D.forward(X))


def test_dense_and_rounded_calls_share_a_workspace():
    L = oracle_layer(*FC2)
    D = DeviceLayer(L)
    g = np.random.Generator(np.random.PCG64(5))
    W = torch.from_numpy(g.standard_normal((L.d_out, L.d_in)) / 55).to(DEV, BF16)
    act8 = fq.FQ_BF16 | fq.FQ_ACT_BITS(8)

    def dense(x, ws):
        y = torch.full((x.shape[0], L.d_out), float("nan"), dtype=BF16, device=DEV)
        fq.fq_dense_forward(x, x.shape[0], L.d_in, W, L.d_out, y, ws, ws.numel())
        assert fq.fq_check(ws) == 0
        return y

    def rounded(x, ws):
        y = torch.full((x.shape[0], L.d_out), float("nan"), dtype=BF16, device=DEV)
        fq.fq_linear_forward(x, x.shape[0], L.d_in, D.T_in, D.C, D.T_out_t, L.d_out, None, y, ws,
                             ws.numel(), act8)
        assert fq.fq_check(ws) == 0
        return y

    need = max(max(fq.fq_dense_workspace_bytes(M, L.d_in, L.d_out),
                   fq.fq_workspace_bytes(M, L.d_in, L.n_in, L.n_out, L.d_out, act8))
               for M in (16, 100, 200))
    ws = _zeros(need)
    for call, M in ((dense, 100), (dense, 200), (rounded, 200), (rounded, 16), (dense, 100),
                    (rounded, 100), (dense, 200)):
        x = torch.from_numpy(activations(*FC2, M)).to(DEV, BF16)
        got = call(x, ws)
        assert torch.isfinite(got).all()
        assert torch.equal(got, call(x, _zeros(need)))
