"""The workspaces of the weight-reconstruction path hold what it uses and no more."""
import pytest

torch = pytest.importorskip("torch")

import paper_2403_06082_gb300 as fq  # noqa: E402


@pytest.mark.parametrize("d_in,n_in,n_out,d_out", [
    (256, 288, 288, 256), (3072, 3392, 848, 768), (4096, 4512, 4512, 4096), (28672, 31552, 9024, 8192)])
def test_reconstruction_needs_the_forward_of_d_in_tokens(d_in, n_in, n_out, d_out):
    assert fq.fq_reconstruct_workspace_bytes(d_in, n_in, n_out, d_out) == \
        fq.fq_workspace_bytes(d_in, d_in, n_in, n_out, d_out, fq.FQ_BF16)


def test_dense_product_without_splits_needs_the_header():
    # 32 tiles of 128 rows x 8 of 256 tokens: no tile is split, nothing lies behind the header
    assert fq.fq_dense_workspace_bytes(2048, 4096, 4096) == 64 * 1024


@pytest.mark.gpu
@pytest.mark.parametrize("M", [1, 100, 300])
def test_nothing_is_written_past_the_workspace(M):
    d_in, n_in, n_out, d_out = 768, 848, 1136, 1024
    g = torch.Generator(device="cuda").manual_seed(M)

    def rnd(*s):
        return torch.randn(*s, generator=g, device="cuda").bfloat16()

    codes = torch.randint(0, 4, (n_out, n_in), generator=g, device="cuda", dtype=torch.uint8)
    scale = torch.full((n_out,), 0.02, device="cuda").half()
    words = torch.empty(fq.fq_packed_words(n_out, n_in), dtype=torch.int32, device="cuda")
    C = fq.fq_pack(codes, scale.view(torch.int16), (scale * -1.5).view(torch.int16), n_out, n_in,
                   words)
    W = torch.empty(d_out, d_in, dtype=torch.bfloat16, device="cuda")
    y = torch.empty(M, d_out, dtype=torch.bfloat16, device="cuda")
    nr = fq.fq_reconstruct_workspace_bytes(d_in, n_in, n_out, d_out)
    nd = fq.fq_dense_workspace_bytes(M, d_in, d_out)
    wr, wd = (torch.zeros(n + 65536, dtype=torch.uint8, device="cuda") for n in (nr, nd))
    wr[nr:] = 0xA5
    wd[nd:] = 0xA5
    fq.fq_reconstruct_weight(rnd(n_in, d_in), C, rnd(d_out, n_out), d_in, d_out, None, W, wr, nr)
    fq.fq_dense_forward(rnd(M, d_in), M, d_in, W, d_out, y, wd, nd)
    assert fq.fq_check(wr) == 0 and fq.fq_check(wd) == 0
    assert (wr[nr:] == 0xA5).all() and (wd[nd:] == 0xA5).all()
    assert torch.isfinite(W).all() and torch.isfinite(y).all()
