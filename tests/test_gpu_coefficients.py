"""fq_coefficients at the edges of its tiles: sizes that are no multiple of a tile, of a K slice or of
a 16-byte load, and both kernels (few and many tiles).  Every element is a chain of K fused
multiply-adds in fp32, so |C - exact| <= gamma_K sum |a b| with gamma_K = K u / (1 - K u), u = 2^-24,
for either product; through both, with |.| entrywise and K = d_in, then d_out:
    |C - exact| <= ((1 + gamma_din) (1 + gamma_dout) - 1) |T_out| |W| |T_in^T|."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2403_06082_gb300 as fq  # noqa: E402

pytestmark = pytest.mark.gpu
U = 2.0 ** -24


@pytest.mark.parametrize("d_out,d_in,n_out,n_in", [
    (1, 1, 1, 1), (17, 33, 19, 35), (64, 64, 65, 127), (130, 62, 257, 129), (66, 129, 2049, 300),
    (1030, 1026, 1153, 1281), (1024, 1028, 1280, 1284), (40, 48, 23100, 60)])
def test_products_at_tile_edges(d_out, d_in, n_out, n_in):
    g = torch.Generator(device="cuda").manual_seed(n_out + n_in)
    W, T_in, T_out = (torch.randn(*s, generator=g, device="cuda")
                      for s in ((d_out, d_in), (n_in, d_in), (n_out, d_out)))
    C = torch.full((n_out, n_in), float("nan"), device="cuda")
    nb = fq.fq_coefficients_workspace_bytes(d_out, n_in)
    ws = torch.full((nb,), 255, dtype=torch.uint8, device="cuda")
    fq.fq_coefficients(W, d_out, d_in, T_in, n_in, T_out, n_out, C, ws, nb)
    Wd, Ti, To = W.double(), T_in.double(), T_out.double()
    exact = To @ (Wd @ Ti.t())
    gam = [k * U / (1 - k * U) for k in (d_in, d_out)]
    bound = ((1 + gam[0]) * (1 + gam[1]) - 1) * (To.abs() @ (Wd.abs() @ Ti.abs().t()))
    assert ((C.double() - exact).abs() <= bound + 1e-30).all()


def test_kernels_agree_bitwise():
    """Rows 0 .. 127 of C by the small tiles alone and as part of a product on the large ones."""
    g = torch.Generator(device="cuda").manual_seed(3)
    d_out, d_in, n_in, n_out = 517, 300, 530, 3000
    W, T_in, T_out = (torch.randn(*s, generator=g, device="cuda")
                      for s in ((d_out, d_in), (n_in, d_in), (n_out, d_out)))
    nb = fq.fq_coefficients_workspace_bytes(d_out, n_in)
    ws = torch.empty(nb, dtype=torch.uint8, device="cuda")
    C = [torch.empty(rows, n_in, device="cuda") for rows in (128, n_out)]
    for c in C:
        fq.fq_coefficients(W, d_out, d_in, T_in, n_in, T_out, c.shape[0], c, ws, nb)
    assert torch.equal(C[0], C[1][:128])
