"""Kernels at the sizes where their tiling can go wrong: tile edges, remainders, the smallest and largest of a range."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def _ctx(*a, **k):
    from paper_2510_05528_b200 import binding as Bd
    return Bd.ArmorContext(*a, device=DEV, **k)


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


@pytest.mark.parametrize("d_in,tokens", [(128, 1), (128, 4095), (256, 63), (384, 65), (640, 1024), (1024, 1025),
                                         (256, 16384 + 77)])
@pytest.mark.parametrize("form", ["plain", "strided", "unaligned_x", "unaligned_h"])
def test_bf16_gram_as_it_lies_in_memory(d_in, tokens, form):
    """X is read where it lies (any leading dimension that is a multiple of 8); a base or leading dimension that TMA does
    not take goes through the staged path; H may start on any 4-byte boundary.  Sums of exact products in fp32: segments
    of 1,024 terms that truncate (2^-23 per 16 terms: below 64 x 2^-23 = 8e-6 of sum |x_i x_j|), then rounded sums."""
    lead = {"plain": d_in, "strided": d_in + 24, "unaligned_x": d_in + 3, "unaligned_h": d_in}[form]
    buf = torch.randn(tokens * lead + 1, device=DEV, generator=_gen(tokens + d_in)).to(torch.bfloat16)
    off = 1 if form == "unaligned_x" else 0
    X = buf[off: off + tokens * lead].view(tokens, lead)[:, :d_in]
    ctx = _ctx(128, d_in, 128)
    store = torch.ones(d_in * d_in + 1, device=DEV)
    H = store[1:].view(d_in, d_in) if form == "unaligned_h" else store[:-1].view(d_in, d_in)
    ctx.gram(X, H)
    Xd = X.double()
    err = (H.double() - 1.0 - Xd.t() @ Xd).abs()
    assert torch.equal(H, H.t())
    assert (err <= 8e-6 * (1.0 + Xd.abs().t() @ Xd.abs())).all()
    assert ctx.device_status()[:4] == [0, 0, 0, 0]


@pytest.mark.parametrize("d_out,d_in", [(128, 128), (128, 384), (384, 256), (640, 1152), (1024, 2560)])
@pytest.mark.parametrize("precision", ["FP16X3", "FP32X3", "TF32"])
def test_dense_product_with_h_at_tile_edges(d_out, d_in, precision):
    """W H through one iteration's loss: L = <E H, E> with E = W - A S B at the initialisation, tiles of 256 x 256 cut by
    the matrix's edge, with and without the contraction split over several pairs of CTAs."""
    from paper_2510_05528_b200 import binding as Bd
    g = _gen(d_out + d_in)
    W = torch.randn(d_out, d_in, device=DEV, generator=g)
    X = torch.randn(2 * d_in, d_in, device=DEV, generator=g)
    H = (X.double().t() @ X.double()).float()
    ctx = _ctx(d_out, d_in, 128, precision=getattr(Bd, "PREC_" + precision))
    st = ctx.init(W, H)
    loss = ctx.proxy_loss(st, H).item()
    E = (W - st.S).double()
    ref = ((E @ H.double()) * E).sum().item()
    assert abs(loss - ref) <= (2e-2 if precision == "TF32" else 1e-5) * ref
    assert np.isfinite(ref) and ctx.device_status()[:4] == [0, 0, 0, 0]


@pytest.mark.parametrize("d_out,d_in,d_block", [(128, 128, 128), (384, 512, 128), (512, 256, 256), (4096, 1152, 128),
                                                (19072, 2048, 128),
                                                (256, 3200, 128), (2560, 5120, 128)])   # ragged pieces; one CTA an SM up to 64 tokens
def test_few_token_forward_equals_the_large_batch(d_out, d_in, d_block):
    """The packed layer at every token tile of the split product (16, 32, 64, 128) and beside its edges, against the rows
    of a batch that takes the persistent kernels.  Integer operands: every fp32 sum is exact in any order, so the
    roundings to bf16 are the same and the outputs agree bit for bit."""
    from paper_2510_05528_b200 import binding as Bd
    g = _gen(d_out * 7 + d_in)
    ctx = _ctx(d_out, d_in, d_block)

    def ints(lo, hi, *shape):
        return torch.randint(lo, hi + 1, shape, device=DEV, generator=g).float()
    S = ints(-2, 2, d_out, d_in)
    grp = S.view(d_out, d_in // 4, 4)
    keep = torch.zeros_like(grp, dtype=torch.bool).scatter_(2, torch.rand(grp.shape, device=DEV, generator=g).topk(2, 2).indices, True)
    grp.mul_(keep)
    M = (keep * torch.tensor([1, 2, 4, 8], device=DEV)).sum(2).to(torch.uint8)
    st = Bd.LayerState(Wbar=S, A=ints(-1, 1, d_out // d_block, d_block, d_block), B=ints(-1, 1, d_in // d_block, d_block, d_block),
                       S=S, M=M)
    packed = ctx.pack_layer(st)
    x = ints(-1, 1, 2100, d_in).to(torch.bfloat16)                     # (more than 2,048 tokens: the persistent kernels whatever the size)
    big = ctx.apply_layer(packed, x)
    z1 = torch.einsum("tjk,jmk->tjm", x.float().view(2100, -1, d_block), st.B).reshape(2100, d_in).to(torch.bfloat16)
    z2 = (z1.double() @ S.double().t()).to(torch.bfloat16)
    y = torch.einsum("tjk,jmk->tjm", z2.double().view(2100, -1, d_block), st.A.double()).reshape(2100, d_out).float().to(torch.bfloat16)
    assert torch.equal(big, y)
    for n in (1, 15, 16, 17, 24, 25, 32, 33, 63, 64, 65, 127, 128, 129, 300):
        assert torch.equal(ctx.apply_layer(packed, x[:n].contiguous()), big[:n]), n
    assert ctx.device_status()[:5] == [0, 0, 0, 0, 0]


@pytest.mark.parametrize("d_out,d_in,d_block", [(512, 2048, 128), (4096, 2048, 128), (5120, 1024, 128), (1024, 2048, 256)])
def test_few_token_forward_of_real_numbers_against_fp64(d_out, d_in, d_block):
    """The sums of the packed forward are fp32 however the core's contraction is cut, and z1, z2 and y are rounded to bf16 once.  At most 64
    truncating additions put a sum off by 64 * 2^-24 of itself, so that at most 2 * 64 * 2^-24 / 2^-8 = 2e-3 of the values
    are rounded the other way, by 2^-7 of themselves at most: sqrt(3 * 2e-3) * 2^-7 = 6e-4 in the norm after three roundings.  (Pieces rounded
    to bf16 before they are added: 1.1e-3 and more.)"""
    from paper_2510_05528_b200 import binding as Bd
    g = _gen(d_out + d_in + d_block)
    ctx = _ctx(d_out, d_in, d_block)
    W = torch.randn(d_out, d_in // 4, 4, device=DEV, generator=g)
    keep = torch.zeros_like(W, dtype=torch.bool).scatter_(2, W.abs().topk(2, dim=2).indices, True)
    S = (W * keep).view(d_out, d_in)
    M = (keep * torch.tensor([1, 2, 4, 8], device=DEV)).sum(2).to(torch.uint8)
    A = torch.eye(d_block, device=DEV) + 0.3 / d_block ** 0.5 * torch.randn(d_out // d_block, d_block, d_block, device=DEV, generator=g)
    B = torch.eye(d_block, device=DEV) + 0.3 / d_block ** 0.5 * torch.randn(d_in // d_block, d_block, d_block, device=DEV, generator=g)
    packed = ctx.pack_layer(Bd.LayerState(Wbar=S, A=A, B=B, S=S, M=M))
    A, B, S = (t.to(torch.bfloat16).double() for t in (A, B, S))
    x = (torch.randn(2100, d_in, device=DEV, generator=g) * torch.exp(torch.randn(d_in, device=DEV, generator=g))).to(torch.bfloat16)
    z1 = torch.einsum("tjk,jmk->tjm", x.double().view(2100, -1, d_block), B).reshape(2100, d_in).to(torch.bfloat16)
    z2 = (z1.double() @ S.t()).to(torch.bfloat16)
    y = torch.einsum("tjk,jmk->tjm", z2.double().view(2100, -1, d_block), A).reshape(2100, d_out).to(torch.bfloat16).double()
    for n in (1, 16, 24, 25, 64, 128, 129, 300, 768, 2048, 2100):
        assert (ctx.apply_layer(packed, x[:n].contiguous()).double() - y[:n]).norm() <= 6e-4 * y[:n].norm(), n
    assert ctx.device_status()[:5] == [0, 0, 0, 0, 0]


@pytest.mark.parametrize("d_out,d_in,d_block,tokens", [
    (128, 128, 128, (129, 640, 641, 1024, 1025, 2200)),             # few-token kernels up to 640; whole and ragged boxes of 32 rows; chunks of 1,024
    (128, 384, 128, (1024, 1027)), (384, 128, 128, (1024, 1027)),   # a chunk's z1 and z2 fill their scratch
    (384, 640, 128, (300, 2048, 2049)),            # some token tiles of 128; a row tile a CTA
    (1024, 384, 128, (256, 1536, 1537)),           # 96 tiles of the few-token core product, and one more
    (256, 2304, 256, (250, 400)),                  # few tokens with z1 by either kernel
    (19072, 256, 128, (129, 145)),                 # CTAs that go from one block to the next
    (512, 256, 256, (129, 200, 2100)),             # blocks of 256 in halves
    (4096, 2304, 256, (129, 300, 513, 1300)),      # on either side of that rule's line; whole blocks over several tiles
    (4096, 512, 128, (1152, 1153, 1500, 2000, 2001)),   # core product: two row tiles by 128, 160, 192, 224 tokens, and one
    (768, 512, 128, (2050,)), (2560, 640, 128, (1500, 1700)),   # an odd number of row tiles; odd groups of rows
])
def test_wrapper_products_of_the_packed_forward(d_out, d_in, d_block, tokens):
    """The products on either side of the core beyond the few-token kernels.  Integer operands: every fp32 sum is exact,
    so the bf16 outputs are the oracle's; rows past the last one are not written."""
    from paper_2510_05528_b200 import binding as Bd
    g = _gen(d_out + 3 * d_in)
    ctx = _ctx(d_out, d_in, d_block)

    def ints(lo, hi, *shape):
        return torch.randint(lo, hi + 1, shape, device=DEV, generator=g).float()
    S = ints(-1, 1, d_out, d_in)
    grp = S.view(d_out, d_in // 4, 4)
    keep = torch.zeros_like(grp, dtype=torch.bool).scatter_(2, torch.rand(grp.shape, device=DEV, generator=g).topk(2, 2).indices, True)
    grp.mul_(keep)
    M = (keep * torch.tensor([1, 2, 4, 8], device=DEV)).sum(2).to(torch.uint8)
    st = Bd.LayerState(Wbar=S, A=ints(-1, 1, d_out // d_block, d_block, d_block), B=ints(-1, 1, d_in // d_block, d_block, d_block),
                       S=S, M=M)
    packed = ctx.pack_layer(st)
    for n in tokens:
        x = ints(-1, 1, n, d_in).to(torch.bfloat16)
        z1 = torch.einsum("tjk,jmk->tjm", x.double().view(n, -1, d_block), st.B.double()).reshape(n, d_in).to(torch.bfloat16)
        z2 = (z1.double() @ S.double().t()).to(torch.bfloat16)
        y = torch.einsum("tjk,jmk->tjm", z2.double().view(n, -1, d_block), st.A.double()).reshape(n, d_out).float().to(torch.bfloat16)
        out = torch.full((n + 40, d_out), 7.0, dtype=torch.bfloat16, device=DEV)
        Bd.armor_apply_layer(ctx.ctx, packed, x, out[:n])
        assert torch.equal(out[:n], y), n
        assert (out[n:] == 7.0).all(), n
    assert ctx.device_status()[:5] == [0, 0, 0, 0, 0]


@pytest.mark.parametrize("d_out,d_in,d_block,tokens", [
    (4096, 2048, 128, (1024, 1025, 1152, 1153, 1441, 1729, 2016, 2017)),   # one row tile, two by 128, 160, 192, 224 tokens, one
    (2560, 2304, 256, (1793, 2000, 2241)),         # an odd number of groups of rows; 160 and 192 tokens
    (5120, 2048, 128, (769, 1345, 1568)),
])
def test_packed_core_with_fp32_wrappers_at_every_width_of_a_tile(d_out, d_in, d_block, tokens):
    """The core product on the sparse tensor cores with its output in fp32, one and two row tiles to a stage's tokens, ragged.  Integers
    small enough for the wrappers' one tf32 pass (11 bits) and every sum: the outputs are the oracle's, rows past the last are not written."""
    from paper_2510_05528_b200 import binding as Bd
    g = _gen(d_out + d_in)
    ctx = _ctx(d_out, d_in, d_block)

    def turned(n):
        # one entry in every row and column of a block, -2 .. 2 without 0
        v = (torch.randint(1, 3, (n // d_block, d_block), device=DEV, generator=g) * (2 * torch.randint(0, 2, (n // d_block, d_block), device=DEV, generator=g) - 1)).float()
        at = torch.rand(n // d_block, d_block, device=DEV, generator=g).argsort(1)
        return torch.zeros(n // d_block, d_block, d_block, device=DEV).scatter_(2, at[:, :, None], v[:, :, None])
    grp = torch.randint(-1, 2, (d_out, d_in // 4, 4), device=DEV, generator=g).float()
    keep = torch.zeros_like(grp, dtype=torch.bool).scatter_(2, torch.rand(grp.shape, device=DEV, generator=g).topk(2, 2).indices, True)
    S = (grp * keep).view(d_out, d_in)
    M = (keep * torch.tensor([1, 2, 4, 8], device=DEV)).sum(2).to(torch.uint8)
    st = Bd.LayerState(Wbar=S, A=turned(d_out), B=turned(d_in), S=S, M=M)
    packed = ctx.pack_core(st)
    for n in tokens:
        x = (torch.randint(-1, 2, (n, d_in), device=DEV, generator=g) * (torch.rand(n, d_in, device=DEV, generator=g) < 0.2)).to(torch.bfloat16)
        z = torch.einsum("tjk,jmk->tjm", x.double().view(n, -1, d_block), st.B.double()).reshape(n, d_in) @ S.double().t()
        assert z.abs().max() < 2048
        y = torch.einsum("tjk,jmk->tjm", z.view(n, -1, d_block), st.A.double()).reshape(n, d_out).float().to(torch.bfloat16)
        out = torch.full((n + 40, d_out), 7.0, dtype=torch.bfloat16, device=DEV)
        Bd.armor_apply_packed(ctx.ctx, st.A, st.B, packed, None, None, x, out[:n])
        assert torch.equal(out[:n], y), n
        assert (out[n:] == 7.0).all(), n
    assert ctx.device_status()[:5] == [0, 0, 0, 0, 0]


@pytest.mark.parametrize("d_out,d_in,d_block", [(32, 64, 32), (96, 256, 32), (256, 256, 32), (320, 128, 64), (120, 200, 8),
                                                (48, 144, 16), (1024, 512, 64), (160, 96, 32)])
@pytest.mark.parametrize("side", [0, 1])
@pytest.mark.parametrize("transpose", [0, 1])
def test_small_wrapper_products(d_out, d_in, d_block, side, transpose):
    """Products with small wrapper blocks (32 x 32 tiles on fp32 lanes), plain and with an addend, in every operand order;
    an fp32 sum of d_block terms: below d_block * 2^-24 of the sum of magnitudes, plus the addend's rounding."""
    from paper_2510_05528_b200 import binding as Bd
    g = _gen(d_out + 3 * d_in + d_block)
    ctx = _ctx(d_out, d_in, d_block, precision=Bd.PREC_SIMT, h_mode=Bd.H_DIAG)
    X = torch.randn(d_out, d_in, device=DEV, generator=g)
    D = torch.randn(d_out, d_in, device=DEV, generator=g)
    nb = (d_out if side else d_in) // d_block
    Q = torch.randn(nb, d_block, d_block, device=DEV, generator=g)
    Qd = (Q.transpose(1, 2) if transpose else Q).double()
    if side:
        ref = (Qd @ X.double().view(nb, d_block, d_in)).view(d_out, d_in)
        mag = (Qd.abs() @ X.double().abs().view(nb, d_block, d_in)).view(d_out, d_in)
    else:
        ref = torch.einsum("rjk,jkm->rjm", X.double().view(d_out, nb, d_block), Qd).reshape(d_out, d_in)
        mag = torch.einsum("rjk,jkm->rjm", X.double().abs().view(d_out, nb, d_block), Qd.abs()).reshape(d_out, d_in)
    out = torch.empty_like(X)
    Bd.armor_block_product(ctx.ctx, side, transpose, Q, X, out, 1.0, None, 0.0, 0)
    assert ((out.double() - ref).abs() <= d_block * 2.0 ** -24 * mag + 1e-30).all()
    Bd.armor_block_product(ctx.ctx, side, transpose, Q, X, out, -1.0, D, 1.0, 0)
    assert ((out.double() - (D.double() - ref)).abs() <= (d_block + 2) * 2.0 ** -24 * (mag + D.double().abs())).all()


@pytest.mark.parametrize("d_block,nb_out,nb_in", [(32, 8, 5), (64, 2, 9), (96, 3, 2), (128, 2, 3), (128, 40, 2), (128, 80, 1),
                                                  (160, 2, 1), (192, 1, 2), (224, 2, 2), (256, 2, 3)])
def test_block_solves(d_block, nb_out, nb_in):
    """A-step and B-step of one iteration with the diagonal weighting, for every panel count and every number of right-hand
    sides per warp: A - I solves (T D T^T + lam I) and the losses only fall.  fp32 solve of systems whose condition number
    is below 1e3 by construction (d_in rows of T exceed d_block): 1e-4 of the result."""
    from paper_2510_05528_b200 import binding as Bd
    d_out, d_in = nb_out * d_block, nb_in * d_block * 4
    g = _gen(d_block + nb_out)
    W = torch.randn(d_out, d_in, device=DEV, generator=g)
    h = torch.rand(d_in, device=DEV, generator=g) + 0.5
    H = torch.diag(h)
    ctx = _ctx(d_out, d_in, d_block, precision=Bd.PREC_FP16X3, h_mode=Bd.H_DIAG, phases=1)   # A-step alone
    st = ctx.init(W, H)
    A0, S0 = st.A.clone(), st.S.clone()
    stats = ctx.read_stats(ctx.bcd_step(st, H, 0, 1))
    T = S0.double().view(nb_out, d_block, d_in)
    E = (W - S0).double().view(nb_out, d_block, d_in)
    G = (T * h.double()) @ T.transpose(1, 2)
    lam = 1e-6 * G.diagonal(dim1=1, dim2=2).sum(1) / d_block
    rhs = (E * h.double()) @ T.transpose(1, 2)
    Gl = G + lam[:, None, None] * torch.eye(d_block, device=DEV, dtype=torch.float64)
    X = torch.linalg.solve(Gl, rhs.transpose(1, 2)).transpose(1, 2)
    assert torch.linalg.cond(Gl).max() < 1e3
    got = (st.A - A0).double()
    assert (got - X).norm() <= 1e-4 * X.norm()
    dec = (rhs * X).sum() + (lam[:, None, None] * X * X).sum()
    assert abs((stats["loss_start"][0] - stats["loss_A"][0]) - dec.item()) <= 1e-3 * dec.item()
    assert ctx.device_status()[:4] == [0, 0, 0, 0]


@pytest.mark.parametrize("n_keep,m_group", [(2, 4), (4, 8), (6, 8)])
@pytest.mark.parametrize("mode", ["diag", "full"])
@pytest.mark.parametrize("d_out,d_in", [(128, 128), (384, 256), (2688, 1024)])
def test_core_step_with_the_mask_applied_in_the_gradient(n_keep, m_group, mode, d_out, d_in):
    """S-step alone from a state off the initialisation: S moves along Gamma (.) M by |Gamma_M|^2 / tr(V H V^T), the other
    entries stay zero.  Three-pass products of 128 terms behind one with d_in terms: 2e-5 of the move."""
    from paper_2510_05528_b200 import binding as Bd
    db = 128
    g = _gen(d_out + d_in + m_group)
    W = torch.randn(d_out, d_in, device=DEV, generator=g)
    X = torch.randn(2 * d_in, d_in, device=DEV, generator=g)
    H = torch.diag(torch.rand(d_in, device=DEV, generator=g) + 0.5) if mode == "diag" else (X.double().t() @ X.double()).float()
    ctx = _ctx(d_out, d_in, db, n_keep=n_keep, m_group=m_group, phases=4, h_mode=Bd.H_DIAG if mode == "diag" else Bd.H_FULL)
    st = ctx.init(W, H)
    st.A.add_(torch.randn(st.A.shape, device=DEV, generator=g) * 0.05)
    st.B.add_(torch.randn(st.B.shape, device=DEV, generator=g) * 0.05)
    S0 = st.S.clone()
    keep = torch.stack([(st.M.int() >> k) & 1 for k in range(m_group)], -1).view(d_out, d_in).bool()
    Ad, Bd64 = torch.block_diag(*st.A.double()), torch.block_diag(*st.B.double())
    Hd = H.double()
    Gm = (Ad.t() @ (W.double() - Ad @ S0.double() @ Bd64) @ Hd @ Bd64.t()) * keep
    V = Ad @ Gm @ Bd64
    tau = (Gm * Gm).sum() / ((V @ Hd) * V).sum()
    ctx.bcd_step(st, H, 0, 1)
    move = (st.S - S0).double()
    assert (st.S[~keep] == 0).all()
    assert (move - tau * Gm).norm() <= 2e-5 * (tau * Gm).norm() + 2.0 ** -24 * S0.double().norm()
    assert ctx.device_status()[:4] == [0, 0, 0, 0]


@pytest.mark.parametrize("m_group,n_keep", [(4, 2), (8, 4), (8, 6)])
def test_initial_mask_orders_scores_as_fp64_does(m_group, n_keep):
    """Scores that fp32 cannot tell apart (equal magnitudes, one ulp apart, products that underflow, overflow or vanish)
    are ordered by their fp64 values, ties to the lower column."""
    d_out, d_in, db = 64, 256, 16
    g = _gen(m_group + n_keep)
    from paper_2510_05528_b200 import binding as Bd
    W = torch.randn(d_out, d_in, device=DEV, generator=g)
    W[8:16] = W[8:16].sign()
    W[16:24] = W[16:24].sign() * torch.nextafter(torch.ones(1, device=DEV), torch.full((1,), 2.0, device=DEV)) ** \
        torch.randint(0, 3, (8, d_in), device=DEV, generator=g).float()
    W[24:32] *= 1e-25
    W[32:40] *= 1e19
    W[40:44] = 0.0
    h = torch.exp(2 * torch.randn(d_in, device=DEV, generator=g))
    h[:64] = 1.0
    h[64:72] = 0.0
    ctx = _ctx(d_out, d_in, db, precision=Bd.PREC_SIMT, h_mode=Bd.H_DIAG, m_group=m_group, n_keep=n_keep)
    st = ctx.init(W, torch.diag(h))
    sc = (W.double() * W.double() * h.double()).view(d_out, -1, m_group)
    order = torch.argsort(sc, dim=2, descending=True, stable=True)[:, :, :n_keep]
    keep = torch.zeros_like(sc, dtype=torch.bool).scatter_(2, order, True)
    bits = (keep * (1 << torch.arange(m_group, device=DEV))).sum(2).to(torch.uint8)
    assert torch.equal(st.M, bits)


@pytest.mark.parametrize("scale", [1.0, 1e-18, 1e16])
def test_row_norms_of_the_normalisation(scale):
    """r2 is the fp64 norm rounded once (half an ulp, at most 2^-24 of it, and 2^-40 for the sum itself; r1 is taken as stored),
    for widths below and above a CTA's stride, with a zero row and a zero column."""
    from paper_2510_05528_b200 import binding as Bd
    for d_in in (64, 1024, 4352):
        g = _gen(d_in)
        W = torch.randn(96, d_in, device=DEV, generator=g) * torch.exp(3 * torch.randn(d_in, device=DEV, generator=g)) * scale
        W[5] = 0.0
        W[:, 7] = 0.0
        ctx = _ctx(96, d_in, 32, precision=Bd.PREC_SIMT, h_mode=Bd.H_DIAG, normalize=1)
        st = ctx.init(W, torch.eye(d_in, device=DEV))
        r2 = (W.double() / st.r1.double()).norm(dim=1)
        r2[5] = 1.0
        assert ((st.r2.double() - r2).abs() <= (2.0 ** -24 + 2.0 ** -40) * r2).all()


@pytest.mark.parametrize("rows,cols", [(256, 256), (1025, 512), (4864, 2048), (4801, 2048), (4864, 2052), (2560, 4096)])
@pytest.mark.parametrize("side,transpose", [(0, 0), (0, 1), (1, 0), (1, 1)])
def test_products_with_blocks_of_256_on_pairs_of_ctas(rows, cols, side, transpose):
    """The kernel for pairs of CTAs gives the bits of the streaming kernel (path 1): same operand parts, same order of MMAs; ragged
    rows of a right product and columns of a left one, with an addend, in place.  It takes 148 tiles of 256 x 256 and more
    (the last four shapes); the first two lie below that line and stay with the streaming kernel."""
    from paper_2510_05528_b200 import binding as Bd
    if (cols if side == 0 else rows) % 256:
        pytest.skip("not a shape of this side")
    g = _gen(rows + cols)
    ctx = _ctx(2560, 2048, 256)
    X = torch.randn(rows, cols, device=DEV, generator=g)
    D = torch.randn(rows, cols, device=DEV, generator=g)
    Q = torch.randn((rows if side else cols) // 256, 256, 256, device=DEV, generator=g)
    out = {}
    for path in (1, -1):
        a, b = torch.full_like(X, 7.0), D.clone()
        Bd.armor_block_product(ctx.ctx, side, transpose, Q, X, a, 1.5, None, 0.0, path)
        Bd.armor_block_product(ctx.ctx, side, transpose, Q, X, b, -1.0, b, 1.0, path)
        out[path] = (a, b)
    assert torch.equal(out[1][0], out[-1][0]) and torch.equal(out[1][1], out[-1][1])
    assert ctx.device_status()[:4] == [0, 0, 0, 0]


@pytest.mark.parametrize("d_out,d_in", [(512, 2304), (4864, 2304), (18944, 512)])
def test_dual_product_and_grams_with_blocks_of_256(d_out, d_in):
    """Dual product: the bits of the streaming kernel, the dot product to the order of its fp64 partial sums; the A-step of an
    iteration (both Grams over the row blocks) against fp64.  Pairs of CTAs take the dual product from 148 tiles (the last two
    shapes have 171 and 148) and the Grams from 74 blocks (the last shape); the first shape stays with the streaming kernel."""
    from paper_2510_05528_b200 import binding as Bd
    g = _gen(d_out + d_in)
    ctx = _ctx(d_out, d_in, 256)
    Q = torch.randn(d_out // 256, 256, 256, device=DEV, generator=g) / 16
    X1, X2 = (torch.randn(d_out, d_in, device=DEV, generator=g) for _ in range(2))
    a, b = torch.empty_like(X1), torch.empty_like(X1)
    d1 = Bd.armor_block_product_dual(ctx.ctx, Q, X1, X2, a, path=1)
    d2 = Bd.armor_block_product_dual(ctx.ctx, Q, X1, X2, b, path=-1)
    assert torch.equal(a, b)
    V1, V2 = (torch.matmul(Q.double(), X.double().view(-1, 256, d_in)) for X in (X1, X2))
    for d in (d1, d2):
        assert abs(d - (V1 * V2).sum().item()) <= 2e-6 * (V1.norm() * V2.norm()).item()
    # A-step alone with the diagonal weighting: X = E D T^T (T D T^T + lam I)^-1 per row block
    h = torch.rand(d_in, device=DEV, generator=g) + 0.5
    ctx = _ctx(d_out, d_in, 256, h_mode=Bd.H_DIAG, phases=1)
    st = ctx.init(X1, torch.diag(h))
    A0, S0 = st.A.clone().double(), st.S.clone()
    ctx.bcd_step(st, torch.diag(h), 0, 1)
    T, E = (M.double().view(-1, 256, d_in) for M in (S0, X1 - S0))
    G = (T * h.double()) @ T.transpose(1, 2)
    G = G + 1e-6 * G.diagonal(dim1=1, dim2=2).mean(1)[:, None, None] * torch.eye(256, device=DEV, dtype=torch.float64)
    X = torch.linalg.solve(G, ((E * h.double()) @ T.transpose(1, 2)).transpose(1, 2)).transpose(1, 2)
    cond = torch.linalg.cond(G).max().item()
    assert (st.A.double() - A0 - X).norm() <= max(1e-4, 1e-6 * cond) * X.norm()


@pytest.mark.parametrize("d_out,d_in,d_block", [(64, 64, 32), (256, 128, 128), (384, 1280, 128), (512, 256, 256)])
@pytest.mark.parametrize("normalize", [0, 1])
def test_fp32_forward_over_chunk_edges(d_out, d_in, d_block, normalize):
    """y = A S B x in fp32 for token counts below, at and above a chunk (four times the smaller dimension).  Bound: each of the three
    products adds at most 3 x 128 / 8 truncated sums of its wrapper's (the core's: one segment's) accumulator, 48 x 2^-24 =
    2.9e-6 of the result each, beside 2^-21 for the parts left out: 1e-5 in all."""
    from paper_2510_05528_b200 import binding as Bd
    g = _gen(d_out + d_in + normalize)
    W = torch.randn(d_out, d_in, device=DEV, generator=g)
    ctx = _ctx(d_out, d_in, d_block, h_mode=Bd.H_DIAG, normalize=normalize)
    st = ctx.init(W, torch.eye(d_in, device=DEV))
    st.A.add_(torch.randn(st.A.shape, device=DEV, generator=g) * 0.1)
    st.B.add_(torch.randn(st.B.shape, device=DEV, generator=g) * 0.1)
    Wh = torch.block_diag(*st.A.double()) @ st.S.double() @ torch.block_diag(*st.B.double())
    if normalize:
        Wh = st.r2.double()[:, None] * Wh * st.r1.double()[None, :]
    chunk = min(4 * min(d_out, d_in), 16384)
    for n in (1, 3, chunk - 1, chunk, chunk + 1, 2 * chunk + 77):
        x = torch.randn(n, d_in, device=DEV, generator=g)
        y = ctx.apply(st, x, denormalize=bool(normalize)).double()
        ref = x.double() @ Wh.t()
        assert (y - ref).norm() <= 1e-5 * ref.norm(), n
    assert ctx.device_status()[:4] == [0, 0, 0, 0]


@pytest.mark.parametrize("d_in,tokens", [(128, 1), (384, 63), (640, 1025), (256, 16384 + 77)])
@pytest.mark.parametrize("form", ["plain", "strided", "unaligned"])
def test_fp32_gram_staged_as_it_lies(d_in, tokens, form):
    """Three-pass Gram of fp32 activations with channels of very different scales: the staged parts hold 22 bits below a
    channel's largest entry, and a segment of 1,024 tokens is 3 x 64 sums that truncate, each by less than 2^-23 of the running
    sum: (192 x 2^-23 + 2^-21) of the products of the channels' norms."""
    lead = {"plain": d_in, "strided": d_in + 20, "unaligned": d_in + 3}[form]
    g = _gen(tokens + d_in)
    buf = torch.randn(tokens * lead + 1, device=DEV, generator=g)
    off = 1 if form == "unaligned" else 0
    X = buf[off: off + tokens * lead].view(tokens, lead)[:, :d_in]
    X.mul_(torch.exp(4 * torch.randn(d_in, device=DEV, generator=g)))
    ctx = _ctx(128, d_in, 128)
    H = ctx.new_gram()
    ctx.gram(X, H)
    Xd = X.double()
    nrm = Xd.norm(dim=0)
    assert torch.equal(H, H.t())
    assert ((H.double() - Xd.t() @ Xd).abs() <= (192 * 2.0 ** -23 + 2.0 ** -21) * nrm[:, None] * nrm[None, :]).all()


def test_few_token_forward_in_a_captured_graph():
    """The dependent launches of the few-token forward are captured and replayed like any others."""
    from paper_2510_05528_b200 import binding as Bd
    d_out, d_in = 1024, 768
    g = _gen(3)
    ctx = _ctx(d_out, d_in, 128)
    W = torch.randn(d_out, d_in, device=DEV, generator=g)
    st = ctx.init(W, torch.eye(d_in, device=DEV))
    packed = ctx.pack_layer(st)
    for n in (1, 50, 300):
        x = torch.randn(n, d_in, device=DEV, generator=g).to(torch.bfloat16)
        want = ctx.apply_layer(packed, x).clone()
        y = torch.zeros_like(want)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            Bd.armor_apply_layer(ctx.ctx, packed, x, y)
        for _ in range(3):
            y.zero_()
            graph.replay()
            torch.cuda.synchronize()
            assert torch.equal(y, want), n
        del graph
    assert ctx.device_status()[:4] == [0, 0, 0, 0]


@pytest.mark.parametrize("d_block,d_in,draws", [(4, 1024, 8), (4, 1152, 8), (32, 1024, 4), (128, 1280, 1), (4, 6272, 8)])
def test_carried_product_over_many_column_blocks_and_draws(d_block, d_in, draws):
    """Group updates alone, from a core that was halved: the carried P = S B H_w takes a row from every draw of every column
    block (up to 12,544 here, on rows that thousands of them share), and the next iteration starts from it.  One call of
    three iterations against three calls, each of which forms P anew: the two differ by the rounding of P, sums of up to
    1,568 rows, sqrt(1568) x 2^-24 = 2.4e-6 of P, and by nothing else (the draws cover every group of a small block; the
    masks keep their margins)."""
    from paper_2510_05528_b200 import binding as Bd
    d_out = 128
    g = _gen(d_in + draws)
    W = torch.randn(d_out, d_in, device=DEV, generator=g)
    v = torch.randn(d_in, device=DEV, generator=g)
    H = torch.eye(d_in, device=DEV) + 0.3 * torch.outer(v, v) / v.square().sum()
    got = {}
    for calls in (1, 3):
        ctx = _ctx(d_out, d_in, d_block, mask_groups=draws, phases=8, seed=3)
        st = ctx.init(W, H)
        st.S.mul_(0.5)
        acc = []
        for t in range(calls):
            acc.append(ctx.read_stats(ctx.bcd_step(st, H, t * (3 // calls), 3 // calls)))
        assert acc[0]["mask_accepted"][0] == 1 and acc[0]["delta_L_mask"][0] < 0
        loss = ctx.proxy_loss(st, H).item()
        assert abs(acc[-1]["loss_mask"][-1] - loss) <= 1e-5 * loss
        assert ctx.device_status()[:4] == [0, 0, 0, 0]
        got[calls] = (st.S.clone(), st.M.clone(), loss)
        del ctx, st
    assert torch.equal(got[1][1], got[3][1])
    assert (got[1][0] - got[3][0]).norm() <= 1e-5 * got[3][0].norm()
    assert abs(got[1][2] - got[3][2]) <= 1e-5 * got[3][2]


@pytest.mark.parametrize("tokens", [1000, 4100, 16384 + 3000])
def test_fp32_gram_of_tiny_and_huge_channels(tokens):
    """Channels between 1e-20 and 1e16 side by side, in tiles that are cut along the tokens (256 channels: the only tile) and in
    whole ones (1,000 tokens): every scaling is a power of two, so an entry keeps the accuracy of its channels however
    small they are (the bound of test_fp32_gram_staged_as_it_lies, and 2^-149 where the entry itself is subnormal)."""
    d_in = 256
    g = _gen(tokens)
    scale = 10.0 ** torch.linspace(-20.0, 16.0, d_in, device=DEV, dtype=torch.float64)
    scale = scale[torch.randperm(d_in, device=DEV, generator=g)]
    X = (torch.randn(tokens, d_in, device=DEV, generator=g).double() * scale).float()
    ctx = _ctx(128, d_in, 128)
    H = ctx.new_gram()
    ctx.gram(X, H)
    Xd = X.double()
    nrm = Xd.norm(dim=0)
    err = (H.double() - Xd.t() @ Xd).abs()
    assert torch.isfinite(H).all()
    assert (err <= (192 * 2.0 ** -23 + 2.0 ** -21) * nrm[:, None] * nrm[None, :] + 2.0 ** -149).all()
    assert ctx.device_status()[:4] == [0, 0, 0, 0]


@pytest.mark.parametrize("d_in,tokens", [(32, 1), (96, 129), (160, 1000), (256, 4100), (640, 16384 + 3000), (1056, 127)])
def test_bf16_gram_of_tiny_channels(d_in, tokens):
    """Channels down to 1e-22 beside ordinary ones and channels of zeros, channels that show their size in the last token only,
    and numbers of channels that leave a tile's box, or a CTA's half of it, over the edge.  Bound of
    test_bf16_gram_as_it_lies_in_memory, beside 2^-24 of the product of the channels' norms (sums of multiples of 2^-149
    of channels above 2^-57), and the rounding of an entry that is itself subnormal, once per call."""
    from paper_2510_05528_b200 import binding as Bd
    g = _gen(tokens + d_in)
    sizes = torch.tensor([1.0, 1e-17, 1e-19, 10 ** -20.5, 1e-21, 0.0, 10 ** -21.5, 1e-22], dtype=torch.float64, device=DEV)
    scale = sizes[torch.randint(0, 8, (d_in,), device=DEV, generator=g)]
    X = (torch.randn(tokens, d_in, device=DEV, generator=g).double() * scale).to(torch.bfloat16)
    X[:, 3], X[-1, 3] = 0.0, 1e-19
    X[:, 5], X[-1, 5] = X[:, 5] * 0.0 + 1e-21, 1.0
    ctx = _ctx(128, d_in, 32, h_mode=Bd.H_DIAG)
    H = ctx.new_gram()
    ctx.gram(X, H)
    Xd = X.double()
    nrm = Xd.norm(dim=0)
    ref = Xd.t() @ Xd
    assert torch.equal(H, H.t())
    assert ((H.double() - ref).abs() <= 8e-6 * (Xd.abs().t() @ Xd.abs()) + 2.0 ** -24 * nrm[:, None] * nrm[None, :] + 2.0 ** -149).all()
    ctx.gram(X, H)                       # on top of what is there
    assert ((H.double() - 2 * ref).abs() <= 2 * (8e-6 * (Xd.abs().t() @ Xd.abs()) + 2.0 ** -24 * nrm[:, None] * nrm[None, :] + 2.0 ** -149)).all()
    assert ctx.device_status()[:4] == [0, 0, 0, 0]


@pytest.mark.parametrize("bad", [float("inf"), float("nan")])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("d_in,tokens,at", [(96, 65, 64), (640, 5000, 17), (256, 16384 + 9, 16384 + 8)])
def test_gram_with_a_value_that_is_not_finite(d_in, tokens, at, dtype, bad):
    """One Inf or NaN stays in its channel's row and column and is visible there; the other entries are those of the clean X."""
    from paper_2510_05528_b200 import binding as Bd
    g = _gen(tokens + d_in)
    X = torch.randn(tokens, d_in, device=DEV, generator=g).to(dtype)
    ctx = _ctx(128, d_in, 32, h_mode=Bd.H_DIAG)
    clean, H = ctx.new_gram(), ctx.new_gram()
    ctx.gram(X, clean)
    k = d_in // 3
    X[at, k] = bad
    ctx.gram(X, H)
    others = torch.arange(d_in, device=DEV) != k
    assert not torch.isfinite(H[k, k])
    assert not torch.isfinite(H[k]).any() and not torch.isfinite(H[:, k]).any()
    assert torch.equal(H[others][:, others], clean[others][:, others])


@pytest.mark.parametrize("d_out,d_in,d_block", [(128, 128, 128), (160, 96, 32), (640, 2560, 128), (1024, 6144, 256), (4096, 4096, 128),
                                                (19072, 2048, 128)])
def test_bf16_forward_of_few_tokens_with_the_dense_core(d_out, d_in, d_block):
    """Token counts at the edges of the narrow tiles (32, 64, .. per tile, one tile up to 256, two up to 512, whole tiles beyond),
    core products cut along d_in and not.  Integer operands: every fp32 sum is exact in any order and every value on the way
    is an integer below 2^8 or rounded to bf16 in one place, so the result is that of fp64, bit for bit."""
    from paper_2510_05528_b200 import binding as Bd
    g = _gen(d_out + 5 * d_in)
    ctx = _ctx(d_out, d_in, d_block, h_mode=Bd.H_DIAG)

    def sparse_ints(hi, density, *shape):
        return torch.randint(-hi, hi + 1, shape, device=DEV, generator=g).float() * (torch.rand(shape, device=DEV, generator=g) < density)
    S = sparse_ints(3, 0.5, d_out, d_in)
    A = sparse_ints(1, 4.0 / d_block, d_out // d_block, d_block, d_block)
    B = sparse_ints(1, 4.0 / d_block, d_in // d_block, d_block, d_block)
    st = Bd.LayerState(Wbar=S, A=A, B=B, S=S, M=torch.zeros(d_out, d_in // 4, dtype=torch.uint8, device=DEV))
    x = sparse_ints(2, 0.5, 600, d_in).to(torch.bfloat16)
    z1 = torch.einsum("tjk,jmk->tjm", x.double().view(600, -1, d_block), B.double()).reshape(600, d_in)
    assert z1.abs().max() < 256
    z2 = z1 @ S.double().t()
    assert z2.abs().max() < 2 ** 11                      # exact as one tf32 operand of the last product
    y = torch.einsum("tjk,jmk->tjm", z2.view(600, -1, d_block), A.double()).reshape(600, d_out).float().to(torch.bfloat16)
    for n in (1, 2, 31, 32, 33, 64, 65, 127, 128, 129, 224, 225, 255, 256, 257, 300, 448, 449, 511, 512, 513, 600):
        assert torch.equal(ctx.apply(st, x[:n].contiguous()), y[:n]), n
    assert ctx.device_status()[:4] == [0, 0, 0, 0]


@pytest.mark.parametrize("precision", ["FP16X3", "FP32X3"])
@pytest.mark.parametrize("d_out,d_in", [(256, 512), (4096, 4096)])
def test_fused_dot_product_keeps_small_terms(d_out, d_in, precision):
    """L = <E H, E> of an E with rows of 1024 and rows of 7 / 16 in turns of 16, H = I: every product and every sum of the 16
    terms that a lane adds in fp32 is exact (2^20 or 49 / 256 each), and a lane's two runs meet in fp64.  Summed in fp32 across
    the runs the small rows vanish (2^24 + 0.77), 1.8e-7 of the loss."""
    from paper_2510_05528_b200 import binding as Bd
    ctx = _ctx(d_out, d_in, 128, precision=getattr(Bd, "PREC_" + precision))
    W = torch.full((d_out, d_in), 1024.0, device=DEV)
    W.view(-1, 2, 16, d_in)[:, 1] = 0.4375
    H = torch.eye(d_in, device=DEV)
    st = ctx.init(W, H)
    st.S.zero_()
    loss = ctx.proxy_loss(st, H).item()
    ref = W.double().square().sum().item()
    assert abs(loss - ref) <= 1e-9 * ref
    assert ctx.device_status()[:4] == [0, 0, 0, 0]


@pytest.mark.parametrize("d_out,d_in", [(768, 18944), (1024, 19200), (768, 2560)])
def test_column_grams_with_blocks_of_256(d_out, d_in):
    """B-step of one iteration with the diagonal weighting, its two Grams over the column blocks in one launch (streaming kernel) and
    one by one (armor_fuse_grams off), where pairs of CTAs take them from 74 blocks on (the first two shapes): C_j = U_j^T U_j
    and Gamma_j = U_j^T (E H)_j through the direction (C_j + lam I)^-1 Gamma_j (H_jj + mu I)^-1, against fp64.  fp32 solves of
    systems whose condition number stays below 1e4: 1e-4 of the direction; both forms round alike, so B agrees to 1e-5."""
    from paper_2510_05528_b200 import binding as Bd
    db = 256
    g = _gen(d_out + d_in)
    W = torch.randn(d_out, d_in, device=DEV, generator=g)
    h = torch.rand(d_in, device=DEV, generator=g) + 0.5
    H = torch.diag(h)
    moved = {}
    for fused in (1, 0):
        ctx = _ctx(d_out, d_in, db, h_mode=Bd.H_DIAG, phases=2)
        Bd.armor_fuse_grams(ctx.ctx, bool(fused))
        st = ctx.init(W, H)
        B0, S0 = st.B.clone(), st.S.clone()
        ctx.bcd_step(st, H, 0, 1)
        moved[fused] = (st.B - B0).double()
        assert ctx.device_status()[:4] == [0, 0, 0, 0]
        del ctx, st
    del H
    U = S0.double().view(d_out, -1, db).transpose(0, 1)
    E = (W - S0).double().view(d_out, -1, db).transpose(0, 1)
    hd = h.double().view(-1, 1, db)
    C = U.transpose(1, 2) @ U
    C = C + 1e-6 * C.diagonal(dim1=1, dim2=2).mean(1)[:, None, None] * torch.eye(db, device=DEV, dtype=torch.float64)
    assert torch.linalg.cond(C).max() < 1e4
    D = torch.linalg.solve(C, U.transpose(1, 2) @ (E * hd)) / (hd + 1e-6 * hd.mean(2, keepdim=True))
    for got in moved.values():
        tau = (got * D).sum() / (D * D).sum()
        assert abs(tau - 1.0) < 1e-3 and (got - tau * D).norm() <= 1e-4 * D.norm()
    assert (moved[1] - moved[0]).norm() <= 1e-5 * moved[1].norm()


@pytest.mark.parametrize("nb_out", [37, 38, 75, 112])
def test_solves_of_256_in_several_slices_a_cta(nb_out):
    """More blocks of 256 than a wave of CTAs takes in four slices: two slices or four to a CTA, one factorisation each."""
    test_block_solves(256, nb_out, 1)


@pytest.mark.parametrize("nb_in", [37, 38, 75])
def test_left_solves_of_256_in_several_slices_a_cta(nb_in):
    """The B-step's solve and the inverse of H_jj with the diagonal weighting: B - I = (S_j^T S_j + lam I)^-1 Gamma_j (D_j + mu I)^-1.
    fp32 solves of systems whose condition number is below 1e3: 1e-4 of the result."""
    from paper_2510_05528_b200 import binding as Bd
    db, d_out = 256, 2048
    d_in = nb_in * db
    g = _gen(nb_in)
    W = torch.randn(d_out, d_in, device=DEV, generator=g)
    h = torch.rand(d_in, device=DEV, generator=g) + 0.5
    H = torch.diag(h)
    ctx = _ctx(d_out, d_in, db, h_mode=Bd.H_DIAG, phases=2)   # B-step alone
    st = ctx.init(W, H)
    S = st.S.double().view(d_out, nb_in, db).transpose(0, 1)
    E = (W - st.S).double().view(d_out, nb_in, db).transpose(0, 1)
    D = h.double().view(nb_in, 1, db)
    ctx.bcd_step(st, H, 0, 1)
    eye = torch.eye(db, device=DEV, dtype=torch.float64)
    C = S.transpose(1, 2) @ S
    C = C + 1e-6 * C.diagonal(dim1=1, dim2=2).mean(1)[:, None, None] * eye
    assert torch.linalg.cond(C).max() < 1e3
    X = torch.linalg.solve(C, S.transpose(1, 2) @ (E * D)) / (D + 1e-6 * D.mean(2, keepdim=True))
    assert (st.B.double() - eye - X).norm() <= 1e-4 * X.norm()
    assert ctx.device_status()[:4] == [0, 0, 0, 0]


@pytest.mark.parametrize("d_out,d_in,d_block,tokens", [(256, 128, 128, 4800), (256, 256, 256, 4737), (512, 384, 128, 2369), (1280, 1152, 128, 1000),
                                                      (4096, 2048, 128, 297), (2304, 9216, 128, 640), (512, 512, 128, 16384 + 70),
                                                      (128, 256, 128, 5000), (4096, 2048, 128, 295)])
@pytest.mark.parametrize("core", ["2of4", "any"])
def test_fp32_forward_on_the_sparse_tensor_cores(d_out, d_in, d_block, tokens, core):
    """The core product of many tokens runs on the sparse tensor cores: rows of one K tile to several
    segments, ragged tiles of tokens, a second chunk, and the dense product where rows do not come in 256 or tokens are few.  "any": groups
    with every pattern of entries, the dense product again.  Truncating additions, 48 in either wrapper product and 96 in a segment of the core's, of up to
    2^-24: 1.2e-5 of the result.  One token that is not finite spoils its own row and no other."""
    g = _gen(d_out + d_in + tokens)
    ctx = _ctx(d_out, d_in, d_block)
    from paper_2510_05528_b200 import binding as Bd
    A = torch.eye(d_block, device=DEV) + 0.3 / d_block ** 0.5 * torch.randn(d_out // d_block, d_block, d_block, device=DEV, generator=g)
    B = torch.eye(d_block, device=DEV) + 0.3 / d_block ** 0.5 * torch.randn(d_in // d_block, d_block, d_block, device=DEV, generator=g)
    W = torch.randn(d_out, d_in // 4, 4, device=DEV, generator=g)
    if core == "2of4":
        keep = torch.zeros_like(W, dtype=torch.bool).scatter_(2, W.abs().topk(2, dim=2).indices, True)
    else:
        bits = torch.randint(0, 16, (d_out, d_in // 4, 1), device=DEV, generator=g)
        keep = ((bits >> torch.arange(4, device=DEV)) & 1).bool()
    S = (W * keep).view(d_out, d_in)
    st = Bd.LayerState(Wbar=S, A=A, B=B, S=S, M=torch.zeros(d_out, d_in // 4, dtype=torch.uint8, device=DEV))
    x = torch.randn(tokens, d_in, device=DEV, generator=g) * torch.exp(torch.randn(d_in, device=DEV, generator=g))
    y = ctx.apply(st, x)
    z = torch.einsum("njk,jmk->njm", x.double().view(tokens, -1, d_block), B.double()).reshape(tokens, d_in) @ S.double().t()
    ref = torch.einsum("njk,jmk->njm", z.view(tokens, -1, d_block), A.double()).reshape(tokens, d_out)
    assert (y.double() - ref).norm() <= 1.2e-5 * ref.norm()
    x[tokens - 2, 5] = float("inf")
    yi = ctx.apply(st, x)
    assert not torch.isfinite(yi[tokens - 2]).any()
    others = torch.arange(tokens, device=DEV) != tokens - 2
    assert (yi[others] - y[others]).norm() <= 1e-6 * y.norm()
    x[tokens - 2, 5] = 0.0
    assert torch.isfinite(ctx.apply(st, x)).all()
    assert ctx.device_status()[:4] == [0, 0, 0, 0]


@pytest.mark.parametrize("d_out,d_in,d_block,tokens", [(256, 128, 128, 4800), (256, 256, 256, 4737), (512, 512, 128, 16384 + 70)])
@pytest.mark.parametrize("at", [0, -1])
def test_fp32_forward_of_a_core_with_one_group_that_is_not_2_of_4(d_out, d_in, d_block, tokens, at):
    """One group of three entries, in the first or the last row, sends the call to the dense product: the bits of calls of 2,000 tokens,
    which run there anyway (up to 1,024 columns a sum is one segment however the call is cut).  The call after it is sparse again."""
    g = _gen(d_out + d_in)
    ctx = _ctx(d_out, d_in, d_block)
    from paper_2510_05528_b200 import binding as Bd
    A = torch.randn(d_out // d_block, d_block, d_block, device=DEV, generator=g)
    B = torch.randn(d_in // d_block, d_block, d_block, device=DEV, generator=g)
    W = torch.randn(d_out, d_in // 4, 4, device=DEV, generator=g)
    W[:, :, 2:] = 0.0
    x = torch.randn(tokens, d_in, device=DEV, generator=g)
    st = Bd.LayerState(Wbar=W.view(d_out, d_in), A=A, B=B, S=W.view(d_out, d_in), M=torch.zeros(d_out, d_in // 4, dtype=torch.uint8, device=DEV))
    sparse = ctx.apply(st, x)
    W[at, at, 3] = 1.0
    assert torch.equal(ctx.apply(st, x), torch.cat([ctx.apply(st, t) for t in x.split(2000)]))
    W[at, at, 3] = 0.0
    assert torch.equal(ctx.apply(st, x), sparse)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()                                       # which product runs is decided as the graph runs
    with torch.cuda.graph(graph, stream=torch.cuda.Stream()):
        y = ctx.apply(st, x)
    for entry in (1.0, 0.0, 1.0):
        W[at, at, 3] = entry
        graph.replay()
        assert torch.equal(y, ctx.apply(st, x)) and torch.equal(y, sparse) == (entry == 0.0)
    assert ctx.device_status()[:4] == [0, 0, 0, 0]


@pytest.mark.parametrize("d_in", [128, 1152, 4224, 8320])
@pytest.mark.parametrize("bad", [float("inf"), float("nan")])
def test_fp32_forward_with_tokens_that_are_not_finite(d_in, bad):
    """Rows of every form of the split: a token that is not finite comes out as NaN throughout, the others keep their bits."""
    g = _gen(d_in)
    ctx = _ctx(256, d_in, 128)
    from paper_2510_05528_b200 import binding as Bd
    W = torch.randn(256, d_in // 4, 4, device=DEV, generator=g)
    W[:, :, 1:3] = 0.0
    st = Bd.LayerState(Wbar=W.view(256, d_in), A=torch.randn(2, 128, 128, device=DEV, generator=g), B=torch.randn(d_in // 128, 128, 128, device=DEV, generator=g),
                       S=W.view(256, d_in), M=torch.zeros(256, d_in // 4, dtype=torch.uint8, device=DEV))
    x = torch.randn(4800, d_in, device=DEV, generator=g)
    y = ctx.apply(st, x)
    spoiled = [0, 223, 4799]
    x[spoiled, d_in - 1] = bad
    yi = ctx.apply(st, x)
    assert torch.isnan(yi[spoiled]).all()
    rest = torch.ones(4800, dtype=torch.bool, device=DEV)
    rest[spoiled] = False
    assert torch.equal(yi[rest], y[rest])
    assert ctx.device_status()[:4] == [0, 0, 0, 0]
