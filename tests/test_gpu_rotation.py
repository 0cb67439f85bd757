"""The rotations of the structured-frame forward, by themselves: the forward leaves the rotated tokens
v = R^T x and the un-rotated outputs s of y = R s in its workspace, behind the fused kernel's part, so
v is compared with x and y with s.  Factor shapes are those where the kernel can go wrong: odd
factors, rows that are no multiple of four or of a CTA's share, factors too large for shared memory
(the second from a width of 224 on, the first where a token leaves no room for it).

The products are chains of a and b fused multiply-adds in fp32, so what is rounded to bf16 lies, with
gamma_k = k u / (1 - k u) and u = 2^-24, within
    e = ((1 + gamma_a) (1 + gamma_b) (1 + u) - 1) |A| |V| |B|
of the 64-bit value v, and rounding is monotonic: bf16(v - e) <= y <= bf16(v + e)."""
import copy

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2403_06082_gb300 as fq  # noqa: E402

pytestmark = pytest.mark.gpu
BF16 = torch.bfloat16
N = 256          # the trivial frame's size on the side that is not rotated
U = 2.0 ** -24


def _rotation(a, b, seed):
    g = np.random.Generator(np.random.PCG64([a, b, seed]))
    return (a, b, g.standard_normal((a, a)), g.standard_normal((b, b)),
            g.permutation(a * b).astype(np.int64), g.choice((-1.0, 1.0), a * b))


def _packed(rows, cols, g):
    codes = torch.randint(0, 4, (rows, cols), generator=g, device="cuda", dtype=torch.uint8)
    s = torch.full((rows,), 0.02, device="cuda").half()
    words = torch.empty(fq.fq_packed_words(rows, cols), dtype=torch.int32, device="cuda")
    return fq.fq_pack(codes, s.view(torch.int16), (s * -1.5).view(torch.int16), rows, cols, words)


def _factors(F):
    """Q_a and Q_b as the frame holds them (fp32)."""
    def at(ptr, n):
        o = ptr - F.buf.data_ptr()
        return F.buf[o:o + 4 * n * n].view(torch.float32).view(n, n).double()
    return at(F.c.Qa, F.c.a), at(F.c.Qb, F.c.b)


def _run(x, F_in, C, F_out):
    """y, and the rotated tokens and un-rotated outputs of the call (meaningful where rotated)."""
    M = x.shape[0]
    y = torch.full((M, F_out.d), float("nan"), dtype=BF16, device="cuda")
    nb = fq.fq_implicit_workspace_bytes(M, F_in.d, F_in.n, F_out.n, F_out.d)
    ws = torch.zeros(nb, dtype=torch.uint8, device="cuda")
    fq.fq_linear_forward_implicit(x, M, F_in, C, F_out, None, y, ws, nb)
    assert fq.fq_check(ws) == 0
    at = fq.fq_workspace_bytes(M, F_in.d, F_in.n, F_out.n, F_out.d)
    parts = []
    for d in (F_in.d, F_out.d):
        parts.append(ws[at:at + 2 * M * d].view(BF16).view(M, d).double())
        at += -(-2 * M * d // 256) * 256
    return y.double(), parts[0], parts[1]


def _within(y, v, scale, a, b):
    gam = [k * U / (1 - k * U) for k in (a, b)]
    e = ((1 + gam[0]) * (1 + gam[1]) * (1 + U) - 1) * scale
    lo, hi = ((v + s * e).float().to(BF16).double() for s in (-1, 1))
    assert ((lo <= y) & (y <= hi)).all()


@pytest.mark.parametrize("M", [1, 5, 64])
@pytest.mark.parametrize("a,b", [
    (1, 48), (48, 1), (3, 16), (16, 3), (16, 16), (16, 43), (43, 16), (43, 32), (32, 32), (36, 36),
    (32, 64), (33, 80), (64, 86), (86, 128), (128, 160), (128, 172), (128, 224), (329, 128)])
def test_rotation(a, b, M):
    d = a * b
    rot = _rotation(a, b, 0)
    FR, FN = fq.fq_frame_implicit(1, d, d, rot), fq.fq_frame_implicit(1, N, N, None)
    Qa, Qb = _factors(FR)
    perm, signs = (torch.from_numpy(t).cuda() for t in rot[4:])
    g = torch.Generator(device="cuda").manual_seed(M)
    # analysis: v = D vec(Q_a^T V Q_b), V[perm[i]] = x_i
    x = torch.randn(M, d, generator=g, device="cuda").to(BF16)
    _, got, _ = _run(x, FR, _packed(N, d, g), FN)
    V = torch.empty(M, d, dtype=torch.float64, device="cuda")
    V[:, perm] = x.double()
    V = V.view(M, a, b)
    _within(got, (Qa.t() @ V @ Qb).reshape(M, d) * signs,
            (Qa.t().abs() @ V.abs() @ Qb.abs()).reshape(M, d), a, b)
    # synthesis: y = Pi vec(Q_a (D s) Q_b^T)
    x = torch.randn(M, N, generator=g, device="cuda").to(BF16)
    got, _, s = _run(x, FN, _packed(d, N, g), FR)
    S = (s * signs).view(M, a, b)
    _within(got, (Qa @ S @ Qb.t()).reshape(M, d)[:, perm],
            (Qa.abs() @ S.abs() @ Qb.t().abs()).reshape(M, d)[:, perm], a, b)


@pytest.mark.parametrize("M", [1, 17, 64])
def test_layers_that_share_tokens_and_frame(M):
    """Layers of a group with the same tokens and input frame share one rotation: bitwise the group
    whose layers have their own copies, also beside layers that share only one of the two."""
    d, d_out, k = 768, 1024, 53
    F = [fq.fq_frame_implicit(k, 16, d, _rotation(24, 32, s)) for s in (1, 2)]
    F_out = [fq.fq_frame_implicit(71, 16, d_out, _rotation(32, 32, 3 + s)) for s in range(4)]
    g = torch.Generator(device="cuda").manual_seed(M)
    xs = [torch.randn(M, d, generator=g, device="cuda").to(BF16) for _ in range(2)]
    Cs = []
    for _ in range(4):
        codes = torch.randint(0, 4, (71 * 16, k * 16), generator=g, device="cuda", dtype=torch.uint8)
        s = torch.rand(71 * 16, generator=g, device="cuda").half() * 0.02
        words = torch.empty(fq.fq_packed_words(71 * 16, k * 16), dtype=torch.int32, device="cuda")
        Cs.append(fq.fq_pack(codes, s.view(torch.int16), (s * -1.5).view(torch.int16), 71 * 16,
                             k * 16, words))
    use = [(0, 0), (0, 0), (1, 0), (0, 1)]       # (tokens, frame) of each layer

    def run(own):
        ys = [torch.full((M, d_out), float("nan"), dtype=BF16, device="cuda") for _ in use]
        keep = [xs[t].clone() if own else xs[t] for t, _ in use]
        layers = [fq.ImplicitLayer(x, F[f], C, Fo, None, y)
                  for x, (_, f), C, Fo, y in zip(keep, use, Cs, F_out, ys)]
        nb = fq.fq_implicit_group_workspace_bytes(M, layers)
        ws = torch.zeros(nb, dtype=torch.uint8, device="cuda")
        fq.fq_linear_forward_implicit_group(M, layers, ws, nb)
        assert fq.fq_check(ws) == 0
        return ys

    for shared, own in zip(run(False), run(True)):
        assert torch.isfinite(shared).all()
        assert torch.equal(shared, own)


@pytest.mark.parametrize("M", [1, 17])
@pytest.mark.parametrize("a,b", [(24, 32), (33, 80), (16, 43), (36, 36), (40, 34), (128, 224)])
def test_arrays_off_16_byte_boundaries(a, b, M):
    """A frame's factors, permutation and signs may lie at any 4-byte boundary: the same sums in the
    same order, so bitwise the results of the frame as it was built."""
    d = a * b
    F, FN = fq.fq_frame_implicit(1, d, d, _rotation(a, b, 0)), fq.fq_frame_implicit(1, N, N, None)
    moved, keep = copy.copy(F), []
    moved.c = type(F.c).from_buffer_copy(F.c)
    sizes = dict(Qa=a * a, QaT=a * a, Qb=b * b, QbT=b * b, perm=d, iperm=d, signs=d)
    for name, n in sizes.items():
        at = getattr(F.c, name) - F.buf.data_ptr()
        other = torch.zeros(4 * n + 16, dtype=torch.uint8, device="cuda")
        other[4:4 + 4 * n] = F.buf[at:at + 4 * n]
        setattr(moved.c, name, other.data_ptr() + 4)
        keep.append(other)
    g = torch.Generator(device="cuda").manual_seed(M)
    x = torch.randn(M, d, generator=g, device="cuda").to(BF16)
    C = _packed(N, d, g)
    assert all(torch.equal(p, q) for p, q in zip(_run(x, F, C, FN)[:2], _run(x, moved, C, FN)[:2]))
    x = torch.randn(M, N, generator=g, device="cuda").to(BF16)
    C = _packed(d, N, g)
    assert torch.equal(_run(x, FN, C, F)[0], _run(x, FN, C, moved)[0])
