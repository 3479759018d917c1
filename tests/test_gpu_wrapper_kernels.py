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


@pytest.mark.parametrize("tiles_per_sm", [11.9, 12.0])
def test_bf16_forward_on_either_side_of_the_choice(tiles_per_sm):
    """bf16 activations with fp32 wrappers take one tf32 pass per wrapper product, on the streaming kernel whatever their number: the last
    count of row tiles below the three-pass products' line of twelve tiles per SM and the first on it, the last tile ragged.  Integer operands, every sum exact in fp32, one rounding to bf16:
    the bits of fp64."""
    from paper_2510_05528_b200 import binding as Bd
    d, n_sm = 6144, torch.cuda.get_device_properties(0).multi_processor_count
    row_tiles = -(-12 * n_sm // (d // 128)) - (tiles_per_sm < 12)
    n = 128 * row_tiles - 29
    assert (row_tiles * (d // 128) >= 12 * n_sm) == (tiles_per_sm == 12) and n <= d       # (one chunk of tokens)
    g = _gen(row_tiles)

    def sparse_ints(hi, density, *shape):
        return torch.randint(-hi, hi + 1, shape, device=DEV, generator=g).float() * (torch.rand(shape, device=DEV, generator=g) < density)
    S = sparse_ints(3, 0.5, d, d)
    A, B = (sparse_ints(1, 4.0 / 128, d // 128, 128, 128) for _ in range(2))
    x = sparse_ints(2, 0.5, n, d).to(torch.bfloat16)
    z1 = torch.einsum("tjk,jmk->tjm", x.double().view(n, -1, 128), B.double()).reshape(n, d)
    assert z1.abs().max() < 256                          # exact in bf16
    z2 = z1 @ S.double().t()
    assert z2.abs().max() < 2 ** 11                      # exact as one tf32 operand
    y = torch.einsum("tjk,jmk->tjm", z2.view(n, -1, 128), A.double()).reshape(n, d).float().to(torch.bfloat16)
    ctx = _ctx(d, d, 128, h_mode=Bd.H_DIAG)
    st = Bd.LayerState(Wbar=S, A=A, B=B, S=S, M=torch.zeros(d, d // 4, dtype=torch.uint8, device=DEV))
    assert torch.equal(ctx.apply(st, x), y)
    assert ctx.device_status()[:4] == [0, 0, 0, 0]


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_conversions_and_scales_of_every_remainder(dtype):
    """The passes over the activations of a denormalised forward take four elements a thread: token counts at one to five times the
    2,368 x 256 elements of a round, one token on either side.  Integer operands and scales that are powers of two: the bits of fp64."""
    from paper_2510_05528_b200 import binding as Bd
    g = _gen(148)
    d_out, d_in, most = 1024, 4096, 741

    def sparse_ints(hi, density, *shape):
        return torch.randint(-hi, hi + 1, shape, device=DEV, generator=g).float() * (torch.rand(shape, device=DEV, generator=g) < density)
    S = sparse_ints(3, 0.25, d_out, d_in)
    A, B = (sparse_ints(1, 4.0 / 128, d // 128, 128, 128) for d in (d_out, d_in))
    r1, r2 = (torch.exp2(torch.randint(0, 2, (d,), device=DEV, generator=g).float()) for d in (d_in, d_out))
    x = sparse_ints(2, 0.25, most, d_in).to(dtype)
    z1 = torch.einsum("tjk,jmk->tjm", (x.double() * r1).view(most, -1, 128), B.double()).reshape(most, d_in)
    z2 = z1 @ S.double().t()
    assert z1.abs().max() < 256 and z2.abs().max() < 2 ** 11
    y = (torch.einsum("tjk,jmk->tjm", z2.view(most, -1, 128), A.double()).reshape(most, d_out) * r2).to(dtype)
    ctx = _ctx(d_out, d_in, 128, h_mode=Bd.H_DIAG)
    st = Bd.LayerState(Wbar=S, A=A, B=B, S=S, M=torch.zeros(d_out, d_in // 4, dtype=torch.uint8, device=DEV), r1=r1, r2=r2)
    for n in (1, 3, 147, 148, 149, 295, 296, 297, 443, 444, 445, 591, 592, 593, 739, 740, 741):
        assert torch.equal(ctx.apply(st, x[:n].contiguous(), denormalize=True), y[:n]), n
    assert ctx.device_status()[:4] == [0, 0, 0, 0]


@pytest.mark.parametrize("d_out,d_in,d_block", [(128, 128, 128), (256, 640, 128), (1024, 5120, 128), (2560, 1152, 128), (256, 256, 256),
                                                (768, 1280, 256), (2368, 1216, 64), (1216, 2368, 64)])
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


@pytest.mark.parametrize("by_rows", [True, False])
def test_cut_contractions_of_both_tile_sizes(by_rows):
    """Grams of 37 blocks of 64 on the fp32 lanes are 296 tiles (64 threads each), of 36 blocks 288 (256 threads): either way the
    contraction of 1,216 is cut into four pieces of 304, which end inside the 32 and the 128 that are fetched at once.  Both
    kernels add the same terms in the same order, so the blocks that the two layers share get the same wrapper, bit for bit."""
    from paper_2510_05528_b200 import binding as Bd
    g = _gen(37)
    W = torch.randn(2368, 1216, device=DEV, generator=g)
    if not by_rows:
        W = W.t().contiguous()
    out = {}
    for nb in (37, 36):
        w = (W[:64 * nb] if by_rows else W[:, :64 * nb]).contiguous()
        H = torch.eye(w.shape[1], device=DEV)
        ctx = _ctx(*w.shape, 64, h_mode=Bd.H_DIAG, phases=1 if by_rows else 2, ridge=0.1)
        st = ctx.init(w, H)
        rec = ctx.read_stats(ctx.bcd_step(st, H, 0, 1))
        # (the B-step's length is one number for all blocks: the direction alone is compared)
        out[nb] = st.A if by_rows else (st.B - torch.eye(64, device=DEV)) / float(rec["tau_B"][0])
        assert ctx.device_status()[:4] == [0, 0, 0, 0]
    if by_rows:
        assert torch.equal(out[37][:36], out[36])
    else:
        # B = I + tau Delta is rounded at 1, 2^-24, and tau once more
        assert (out[37][:36] - out[36]).abs().max() <= 4 * 2.0 ** -24 * (1 + out[36].abs().max()) / float(rec["tau_B"][0])


@pytest.mark.parametrize("d_out,d_in,d_block", [(32, 32, 32), (20, 64, 16), (256, 256, 64), (256, 1152, 128), (512, 1024, 128), (516, 1536, 128),
                                                (768, 768, 48), (480, 772, 48), (512, 640, 80), (800, 356, 80)])
@pytest.mark.parametrize("side,transpose", [(0, 0), (0, 1), (1, 0), (1, 1)])
def test_small_products_keep_the_order_of_their_sums(d_out, d_in, d_block, side, transpose):
    """256 threads a tile (up to 295 tiles) and 64 (from 296 on: from the fifth shape): contractions of 16, 48 and 80, no multiple of the 128 and the
    32 that are fetched at once, rows and columns that end inside a tile (the shapes of 772 and 356 columns, left products: four
    columns of the last one).  Integers below 2^8 and sums of at most 256 products of them are exact in fp32."""
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


@pytest.mark.parametrize("d_out", [128, 640, 4224, 16384, 16512])
def test_guards_products_of_few_and_many_row_blocks(d_out):
    """The guard's products with H have a row for every row block: 1, 5, 33 (boxes of 32 rows that are not full), 128 (the most the kernel
    with the rows in tensor memory takes) and 129; the two line searches move E H_w on its way through the gradients, by both steps,
    one, or none.  A wrong row, move or sign shows in the tracked loss, which otherwise is the one evaluated from the state (fp32
    sums: 1e-5 of the start, as above)."""
    d_in = 256
    g = _gen(d_out)
    W = torch.randn(d_out, d_in, device=DEV, generator=g)
    X = torch.randn(4 * d_in, d_in, device=DEV, generator=g)
    H = (X.double().t() @ X.double()).float()
    for phases in (15, 15 - 4, 15 - 2, 9):
        ctx = _ctx(d_out, d_in, 128, phases=phases)
        st = ctx.init(W, H)
        rec = ctx.read_stats(ctx.bcd_step(st, H, 0, 3))
        loss = ctx.proxy_loss(st, H).item()
        assert abs(rec["loss_mask"][-1] - loss) <= 1e-5 * rec["loss_start"][0]
        assert np.all(np.diff(rec["loss_mask"]) <= 0)
        assert ctx.device_status()[:4] == [0, 0, 0, 0]


@pytest.mark.parametrize("d_in", [768, 1024, 1536])
def test_cut_and_uncut_grams_have_the_same_bits(d_in):
    """fp32 activations, 16,384 tokens at a time.  One call for two such chunks stages the second beside the contraction of the first:
    no staging memory is idle, the pieces of these channels' tiles (192 to 672 slabs) do not fit the context's own 160 slabs and the
    tiles stay whole.  A call for each chunk has the second staging buffer for slabs and cuts them."""
    g = _gen(d_in)
    ctx = _ctx(128, d_in, 128)
    X = torch.randn(2 * 16384, d_in, device=DEV, generator=g) * torch.exp(torch.randn(d_in, device=DEV, generator=g))
    whole, cut = ctx.new_gram(), ctx.new_gram()
    ctx.gram(X, whole)
    for half in X.split(16384):
        ctx.gram(half, cut)
    assert torch.equal(whole, cut) and whole.abs().min() > 0
    assert ctx.device_status()[:4] == [0, 0, 0, 0]


@pytest.mark.parametrize("d_in,tokens", [(768, 16384), (1024, 5000), (1024, 16384), (1024, 16385), (1536, 9000), (2048, 16384)])
def test_gram_of_few_channels_is_cut_along_the_tokens(d_in, tokens):
    """Tiles cut at segments of 1,024 tokens add up in the order of an uncut tile: the Gram of bf16 activations, which are not
    scaled, has the bits of one call per segment; fp32 activations, scaled per call, are compared with fp64.  The accumulator drops
    what lies below its last bit: of the squares on the diagonal, which make up the norm, up to 2^-24 per addition, 3 x 64 of them in a segment of 1,024
    tokens, 1.15e-5 (the parts' 22 bits add 1e-7; a segment without one of its three products is 4e-5 off)."""
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
    assert (H.double() - ref).norm() <= 1.2e-5 * ref.norm() and torch.equal(H, H.t())
    assert ctx.device_status()[:4] == [0, 0, 0, 0]


@pytest.mark.parametrize("cols", [3068, 3076])
def test_left_product_with_an_addend_on_either_side_of_its_line(cols):
    """An addend moves the line between the kernels to two tiles per SM (288 and 300 tiles here, 148 SMs)."""
    test_one_sided_products_on_either_side_of_the_choice(1, 1536, cols, 0)


@pytest.mark.parametrize("d_out,d_in,d_block", [(128, 128, 128), (384, 640, 128), (1536, 3072, 128), (1536, 3200, 128), (2560, 4096, 128),
                                                (256, 512, 256), (1024, 1280, 256)])
def test_weighted_residual_of_the_diagonal_weighting(d_out, d_in, d_block):
    """E = W - A S B is never stored, its weighted form and the loss leave the product's epilogue: one tile, both kernels on either
    side of their line (two tiles per SM), blocks of 256.  The tensor cores' accumulator truncates: 3 d_block / 8 additions of up to
    2^-24 each in S B and again in A (S B), and the loss is quadratic in E, hence 4 (3 d_block / 8) 2^-24 (1.2e-5 for 128) of it.
    The weighted residual comes back through the gradients of an Adam step: compared with the CUDA-core kernels, whose products are fp32."""
    from paper_2510_05528_b200 import binding as Bd
    g = _gen(d_out + d_in)
    W = torch.randn(d_out, d_in, device=DEV, generator=g)
    h = torch.rand(d_in, device=DEV, generator=g) * 3 + 0.1
    H = torch.diag(h)
    got = {}
    tol = 1.5 * d_block * 2.0 ** -24
    for precision in (Bd.PREC_FP16X3, Bd.PREC_SIMT):
        ctx = _ctx(d_out, d_in, d_block, precision=precision, h_mode=Bd.H_DIAG, ab_step=Bd.AB_ADAM, adam_lr=1e-3, seed=5)
        st = ctx.init(W, H)
        gen = _gen(3)
        st.A.add_(torch.randn(st.A.shape, device=DEV, generator=gen), alpha=0.05)
        st.B.add_(torch.randn(st.B.shape, device=DEV, generator=gen), alpha=0.05)
        loss = ctx.proxy_loss(st, H).item()
        T = torch.einsum("rjk,jkn->rjn", st.S.double().view(d_out, -1, d_block), st.B.double()).reshape(d_out, d_in)
        E = W.double() - torch.einsum("imk,ikn->imn", st.A.double(), T.view(-1, d_block, d_in)).reshape(d_out, d_in)
        ref = (E * E * h.double()).sum().item()
        assert abs(loss - ref) <= tol * ref
        stats = ctx.read_stats(ctx.bcd_step(st, H, 1, 1))
        got[precision] = (st.A.clone(), st.B.clone(), stats["loss_start"][0], stats["loss_A"][0])
        assert ctx.device_status()[:4] == [0, 0, 0, 0]
    a, b = got[Bd.PREC_FP16X3], got[Bd.PREC_SIMT]
    for k in (0, 1):
        assert (a[k] - b[k]).double().norm() <= 1e-4 * b[k].double().norm()
    for k in (2, 3):
        assert abs(a[k] - b[k]) <= 2 * tol * b[k]


@pytest.mark.parametrize("d_out,d_in,d_block", [(128, 128, 128), (384, 640, 128), (1536, 3200, 128), (2560, 4096, 128), (256, 512, 256), (1024, 1280, 256)])
def test_line_search_of_the_core_with_the_diagonal_weighting(d_out, d_in, d_block):
    """The core's step alone: R = Gamma_M B and R diag(h), which with d_block 128 exists in shared memory only; tau = |Gamma_M|^2 / q with
    q = <A R, A R diag(h)> and S += tau Gamma_M, against fp64.  Four wrapper products in a row, each with 3 d_block / 8 truncating additions of up
    to 2^-24; q is quadratic in the last two of them: 6 (3 d_block / 8) 2^-24 of tau, and as much of the move."""
    from paper_2510_05528_b200 import binding as Bd
    g = _gen(d_out + 3 * d_in)
    W = torch.randn(d_out, d_in, device=DEV, generator=g)
    h = torch.rand(d_in, device=DEV, generator=g) * 3 + 0.1
    H = torch.diag(h)
    ctx = _ctx(d_out, d_in, d_block, h_mode=Bd.H_DIAG, phases=4)
    st = ctx.init(W, H)
    st.A.add_(torch.randn(st.A.shape, device=DEV, generator=g), alpha=0.05)
    st.B.add_(torch.randn(st.B.shape, device=DEV, generator=g), alpha=0.05)
    A, B, S = st.A.double(), st.B.double(), st.S.double()
    left = lambda P, X: torch.einsum("imk,ikn->imn", P, X.view(-1, d_block, d_in)).reshape(d_out, d_in)
    right = lambda X, P: torch.einsum("rjk,jkn->rjn", X.view(d_out, -1, d_block), P).reshape(d_out, d_in)
    EH = (W.double() - left(A, right(S, B))) * h.double()
    keep = ((st.M.long()[:, :, None] >> torch.arange(4, device=DEV)) & 1).bool().view(d_out, d_in)
    G = right(left(A.transpose(1, 2), EH), B.transpose(1, 2)) * keep
    V = left(A, right(G, B))
    tau = ((G * G).sum() / (V * V * h.double()).sum()).item()
    stats = ctx.read_stats(ctx.bcd_step(st, H, 0, 1))
    tol = 6 * 3 * d_block / 8 * 2.0 ** -24
    assert abs(stats["tau_S"][0] - tau) <= tol * tau
    move = st.S.double() - S
    assert (move - tau * G).norm() <= tol * (tau * G).norm() + 2.0 ** -24 * S.norm()
    assert ctx.device_status()[:4] == [0, 0, 0, 0]
