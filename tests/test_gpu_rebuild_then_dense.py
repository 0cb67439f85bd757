"""A rebuilt weight read by the product that is enqueued right behind it.  Both calls wait behind a
few milliseconds of other work on the stream, so that the second is queued before the first
starts and its kernel may be launched while the weight is still being written; the weight holds NaN
from before, and the result is bitwise that of the two calls with a synchronization between."""
import pytest

torch = pytest.importorskip("torch")

import paper_2403_06082_gb300 as fq  # noqa: E402

pytestmark = pytest.mark.gpu
BF16 = torch.bfloat16


@pytest.mark.parametrize("d_in,d_out,M", [(768, 3072, 300), (3072, 768, 2048), (2048, 2048, 64)])
def test_product_waits_for_the_rebuilt_weight(d_in, d_out, M):
    n_in, n_out = ((-(-11 * d // 160)) * 16 for d in (d_in, d_out))
    g = torch.Generator(device="cuda").manual_seed(M)

    def rnd(*s):
        return (torch.randn(*s, generator=g, device="cuda") * 0.05).to(BF16)

    codes = torch.randint(0, 4, (n_out, n_in), generator=g, device="cuda", dtype=torch.uint8)
    scale = torch.full((n_out,), 0.02, device="cuda").half()
    words = torch.empty(fq.fq_packed_words(n_out, n_in), dtype=torch.int32, device="cuda")
    C = fq.fq_pack(codes, scale.view(torch.int16), (scale * -1.5).view(torch.int16), n_out, n_in,
                   words)
    T_in, T_out_t, x = rnd(n_in, d_in), rnd(d_out, n_out), rnd(M, d_in)
    W = torch.empty(d_out, d_in, dtype=BF16, device="cuda")
    y = torch.empty(M, d_out, dtype=BF16, device="cuda")
    nr = fq.fq_reconstruct_workspace_bytes(d_in, n_in, n_out, d_out)
    nd = fq.fq_dense_workspace_bytes(M, d_in, d_out)
    wr, wd = (torch.zeros(n, dtype=torch.uint8, device="cuda") for n in (nr, nd))
    busy = rnd(8192, 8192)

    def calls(between):
        W.fill_(float("nan"))
        y.fill_(float("nan"))
        for _ in range(0 if between else 3):
            torch.matmul(busy, busy)
        fq.fq_reconstruct_weight(T_in, C, T_out_t, d_in, d_out, None, W, wr, nr)
        if between:
            torch.cuda.synchronize()
        fq.fq_dense_forward(x, M, d_in, W, d_out, y, wd, nd)
        assert fq.fq_check(wr) == 0 and fq.fq_check(wd) == 0
        return y.clone()

    expect = calls(True)
    assert torch.isfinite(expect).all()
    for _ in range(5):
        assert torch.equal(calls(False), expect)
