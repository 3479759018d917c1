"""Kernels at the edges of their dispatch: Grams of few channels cut along the tokens, per-block Grams, the choice between the two kernels for one-sided
products, the two tile sizes of small products, the solves' panels and the joint update of the carried product."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _ctx(d_out, d_in, d_block, **kw):
    from paper_2510_05528_b200 import binding as Bd
    return Bd.ArmorContext(d_out, d_in, d_block, device=DEV, **kw)


@pytest.mark.parametrize("side,rows,cols", [(0, 128, 128), (0, 1025, 1024), (0, 28280, 1024), (0, 28416, 1024), (1, 128, 132),
                                            (1, 1536, 4604), (1, 1536, 4612)])
@pytest.mark.parametrize("transpose", [0, 1])
def test_one_sided_products_on_either_side_of_the_choice(side, rows, cols, transpose):
    """The library's choice (path -1) gives the bits of both kernels: one tile, ragged in the free dimension, and the last tile
    count below and the first on the lines (148 SMs: 1,776 tiles of a right product, 444 of a left one)."""
    from paper_2510_05528_b200 import binding as Bd
    g = _gen(rows + cols)
    ctx = _ctx(1024, 1024, 128)
    X = torch.randn(rows, cols, device=DEV, generator=g)
    D = torch.randn(rows, cols, device=DEV, generator=g)
    Q = torch.randn((rows if side else cols) // 128, 128, 128, device=DEV, generator=g)
    out = {}
    for path in (1, 2, -1):
        a, b = torch.full_like(X, 7.0), D.clone()
        Bd.armor_block_product(ctx.ctx, side, transpose, Q, X, a, 1.5, None, 0.0, path)
        Bd.armor_block_product(ctx.ctx, side, transpose, Q, X, b, -1.0, b, 1.0, path)
        out[path] = (a, b)
    for path in (2, -1):
        assert torch.equal(out[1][0], out[path][0]) and torch.equal(out[1][1], out[path][1])
    assert ctx.device_status()[:4] == [0, 0, 0, 0]


@pytest.mark.parametrize("d_out,d_in,d_block", [(128, 128, 128), (256, 640, 128), (1024, 5120, 128), (2560, 1152, 128), (256, 256, 256),
                                                (768, 1280, 256)])
@pytest.mark.parametrize("fused", [1, 0])
def test_block_grams(d_out, d_in, d_block, fused):
    """G_i = T_i D T_i^T, Gamma_i = E_i D T_i^T and C_j = U_j^T U_j, Gamma_j = U_j^T E_j D through the steps that they feed: the exact block
    solves of one iteration against fp64.  One chunk of the contraction up to several slabs of it, more items than SMs, both
    Grams in one launch or one by one.  The operands carry
    22 bits.  The eigenvalues of a system lie between the ridge of 0.1 and six times their mean (sums of at least d_block terms: a factor
    of (1 + 1)^2, weights up to 1.5 times the mean), so its condition is below 60 and 60 * 2^-21 = 3e-5 of the result bounds what the
    parts cause: 1e-4."""
    from paper_2510_05528_b200 import binding as Bd
    g = _gen(d_out + d_in)
    W = torch.randn(d_out, d_in, device=DEV, generator=g)
    h = torch.rand(d_in, device=DEV, generator=g) + 0.5
    eye = torch.eye(d_block, device=DEV, dtype=torch.float64)
    Wd, hd = W.double(), h.double()
    ctx = _ctx(d_out, d_in, d_block, h_mode=Bd.H_DIAG, phases=1, ridge=0.1)
    Bd.armor_fuse_grams(ctx.ctx, bool(fused))
    st = ctx.init(W, torch.diag(h))
    S = st.S.double()
    ctx.bcd_step(st, torch.diag(h), 0, 1)
    T, E = S.view(-1, d_block, d_in), (Wd - S).view(-1, d_block, d_in)
    G = (T * hd) @ T.transpose(1, 2)
    G = G + 0.1 * G.diagonal(dim1=1, dim2=2).mean(1)[:, None, None] * eye
    A = eye + torch.linalg.solve(G, (T * hd) @ E.transpose(1, 2)).transpose(1, 2)
    assert (st.A.double() - A).norm() <= 1e-4 * (A - eye).norm()
    ctx = _ctx(d_out, d_in, d_block, h_mode=Bd.H_DIAG, phases=2, ridge=0.1)
    Bd.armor_fuse_grams(ctx.ctx, bool(fused))
    st = ctx.init(W, torch.diag(h))
    ctx.bcd_step(st, torch.diag(h), 0, 1)
    U, E = (M.view(d_out, -1, d_block).transpose(0, 1) for M in (S, Wd - S))      # [block][row][column]
    C = U.transpose(1, 2) @ U
    C = C + 0.1 * C.diagonal(dim1=1, dim2=2).mean(1)[:, None, None] * eye
    hj = hd.view(-1, 1, d_block)
    Gam = U.transpose(1, 2) @ (E * hj)
    mu = 0.1 * hj.mean(2, keepdim=True)
    Delta = torch.linalg.solve(C, Gam) / (hj + mu)
    V = torch.einsum("jrk,jkn->rjn", U, Delta).reshape(d_out, d_in)
    tau = (Gam * Delta).sum() / (V * V * hd).sum()
    assert (st.B.double() - eye - tau * Delta).norm() <= 1e-4 * (tau * Delta).norm()
    assert ctx.device_status()[:4] == [0, 0, 0, 0]


@pytest.mark.parametrize("d_out,d_in,d_block", [(32, 32, 32), (20, 64, 16), (256, 256, 64), (256, 1152, 128), (512, 1024, 128), (516, 1536, 128)])
@pytest.mark.parametrize("side,transpose", [(0, 0), (0, 1), (1, 0), (1, 1)])
def test_small_products_keep_the_order_of_their_sums(d_out, d_in, d_block, side, transpose):
    """256 threads a tile and 64 (from 296 tiles on: the last two shapes), contractions that are no multiple of what is fetched at once,
    rows that end inside a tile: integers below 2^8 and sums of at most 256 products of them are exact in fp32."""
    from paper_2510_05528_b200 import binding as Bd
    if (d_out if side else d_in) % d_block:
        pytest.skip("not a shape of this side")
    g = _gen(d_out + d_in + d_block)
    ctx = _ctx(d_block, d_block, d_block, precision=Bd.PREC_SIMT, h_mode=Bd.H_DIAG)
    X = torch.randint(-128, 128, (d_out, d_in), device=DEV, generator=g).float()
    nb = (d_out if side else d_in) // d_block
    Q = torch.randint(-128, 128, (nb, d_block, d_block), device=DEV, generator=g).float()
    Qd = (Q.transpose(1, 2) if transpose else Q).double()
    ref = ((Qd @ X.double().view(nb, d_block, d_in)).view(d_out, d_in) if side
           else torch.einsum("rjk,jkm->rjm", X.double().view(d_out, nb, d_block), Qd).reshape(d_out, d_in))
    out = torch.full_like(X, 7.0)
    Bd.armor_block_product(ctx.ctx, side, transpose, Q, X, out, 1.0, None, 0.0, 0)
    assert torch.equal(out.double(), ref)
    Bd.armor_block_product(ctx.ctx, side, transpose, Q, X, out, -1.0, out, 1.0, 0)
    assert not out.any()


@pytest.mark.parametrize("d_out,d_in,d_block", [(256, 512, 32), (256, 512, 128)])
def test_carried_product_moves_by_both_steps(d_out, d_in, d_block):
    """T H_w moves by the B-step's and the core step's direction in one pass when both steps run, each on its own otherwise:
    after four iterations the tracked loss is the one evaluated from the state (fp32 sums: 1e-5 of the start)."""
    from paper_2510_05528_b200 import binding as Bd
    g = _gen(d_block)
    W = torch.randn(d_out, d_in, device=DEV, generator=g)
    X = torch.randn(4 * d_in, d_in, device=DEV, generator=g)
    H = (X.double().t() @ X.double()).float()
    for phases in (15, 15 - 4, 15 - 2):
        ctx = _ctx(d_out, d_in, d_block, phases=phases)
        st = ctx.init(W, H)
        rec = ctx.read_stats(ctx.bcd_step(st, H, 0, 4))
        loss = ctx.proxy_loss(st, H).item()
        assert abs(rec["loss_mask"][-1] - loss) <= 1e-5 * rec["loss_start"][0]
        assert np.all(np.diff(rec["loss_mask"]) <= 0)


@pytest.mark.parametrize("d_in,tokens", [(768, 16384), (1024, 5000), (1024, 16384), (1024, 16385), (1536, 9000), (2048, 16384)])
def test_gram_of_few_channels_is_cut_along_the_tokens(d_in, tokens):
    """Tiles cut at segments of 1,024 tokens add up in the order of an uncut tile: the Gram of bf16 activations, which are not
    scaled, has the bits of one call per segment; fp32 activations, scaled per call, those of fp64 to the parts' 22 bits."""
    g = _gen(d_in + tokens)
    ctx = _ctx(128, d_in, 128)
    X = torch.randn(tokens, d_in, device=DEV, generator=g)
    Xb = X.to(torch.bfloat16)
    H, H1 = ctx.new_gram(), ctx.new_gram()
    ctx.gram(Xb, H)
    for r in range(0, tokens, 1024):
        ctx.gram(Xb[r:r + 1024].contiguous(), H1)
    assert torch.equal(H, H1) and torch.equal(H, H.t())
    H.zero_()
    ctx.gram(X, H)
    ref = X.double().t() @ X.double()
    assert (H.double() - ref).norm() <= 3e-5 * ref.norm() and torch.equal(H, H.t())
    assert ctx.device_status()[:4] == [0, 0, 0, 0]
