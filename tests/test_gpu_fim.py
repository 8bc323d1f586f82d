"""GPU parity of the projected FIM, its damped Cholesky solve and the preconditioned score."""
import numpy as np
import pytest
import torch

from parity import check_close

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    import paper_2505_18976_b200 as g
    g.lib()
    return g


def _compressed(n, k, seed, scale=1.0):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    # correlated columns so that F is far from a multiple of the identity
    Z = torch.randn((n, k), generator=g, device="cuda")
    mix = torch.randn((k, k), generator=g, device="cuda") / k ** 0.5
    return ((Z + 0.5 * Z @ mix) * scale).contiguous()


@pytest.mark.parametrize("n,k", [(1000, 96), (77, 130), (4096, 256), (33, 1), (3000, 520)])
def test_fim_parity(G, oracle_mod, n, k):
    X = _compressed(n, k, 3 + k)
    F = G.grass_fim(X).cpu().numpy()
    ref, absum = oracle_mod.fim(X.cpu().numpy())
    check_close(F, ref, absum, 1e-4, n + 64, eps=2.0 ** -23, what=f"fim n={n} k={k}")
    # mirrored entries get the same addends, possibly in another order across sample chunks
    assert np.all(np.abs(F - F.T) <= 2.0 ** -21 * absum)


def test_fim_of_a_column_slice(G, oracle_mod):
    """One layer's block of a wider compressed matrix (block-diagonal FIM)."""
    X = _compressed(500, 300, 9)
    blk = X[:, 100:228]
    F = G.grass_fim(blk).cpu().numpy()
    ref, absum = oracle_mod.fim(np.ascontiguousarray(blk.cpu().numpy()))
    check_close(F, ref, absum, 1e-4, 564, eps=2.0 ** -23, what="fim column slice")


@pytest.mark.parametrize("n,k,lam,M", [(600, 64, 1e-2, 5), (900, 200, 1e-1, 70), (2000, 333, 1e-2, 256), (50, 100, 0.5, 3)])
def test_factor_and_apply_parity(G, oracle_mod, n, k, lam, M):
    X = _compressed(n, k, 20 + k)
    B = _compressed(M, k, 21 + k)
    F = G.grass_fim(X)
    Fh = F.cpu().numpy().astype(np.float64)
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    L = G.grass_fim_factor(F.clone(), lam, dev_status=st)
    sol = G.grass_fim_apply(L, B.clone()).cpu().numpy().astype(np.float64)
    assert int(st.item()) == 0
    # the factor itself: L L^T = F + lam I
    Lh = np.tril(L.cpu().numpy().astype(np.float64))
    Mh = Fh + lam * np.eye(k)
    assert np.abs(Lh @ Lh.T - Mh).max() <= 1e-5 * np.abs(Mh).max()
    # the solution against the oracle on the same matrix, within the conditioning of the system
    ref = oracle_mod.fim_solve(Fh, lam, B.cpu().numpy().astype(np.float64))
    cond = np.linalg.cond(Mh)
    err = np.linalg.norm(sol - ref, axis=1) / np.linalg.norm(ref, axis=1)
    assert err.max() <= 64 * cond * 2.0 ** -24, (err.max(), cond)
    # and against the oracle chain from the raw data (fim in double, then solve)
    ref2 = oracle_mod.fim_solve(oracle_mod.fim(X.cpu().numpy())[0], lam, B.cpu().numpy().astype(np.float64))
    err2 = np.linalg.norm(sol - ref2, axis=1) / np.linalg.norm(ref2, axis=1)
    assert err2.max() <= 64 * cond * 2.0 ** -23


def test_not_positive_definite_is_flagged(G):
    F = torch.zeros(70, 70, device="cuda")
    F[0, 0] = -1.0
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    G.grass_fim_factor(F, 0.0, dev_status=st)
    torch.cuda.synchronize()
    assert int(st.item()) == G.binding.DEV_NOT_PD


def test_pivots_that_are_not_positive_count_as_one(G):
    F = torch.zeros(140, 140, device="cuda")
    F[3, 3], F[70, 70], F[80, 80] = -1.0, 4.0, 9.0
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    G.grass_fim_factor(F, 0.0, dev_status=st)
    want = torch.ones(140, device="cuda")
    want[70], want[80] = 2.0, 3.0
    assert int(st.item()) == G.binding.DEV_NOT_PD
    assert torch.equal(torch.tril(F), torch.diag(want))


def test_preconditioned_score(G, oracle_mod):
    """scores[i, m] = <g_i, (F + lam I)^-1 g_test,m> through grass_fim -> factor -> apply -> grass_score."""
    n, k, M, lam = 1500, 192, 40, 5e-2
    train = _compressed(n, k, 50)
    test = _compressed(M, k, 51)
    L = G.grass_fim_factor(G.grass_fim(train), lam)
    pt = G.grass_fim_apply(L, test.clone())
    sc = G.grass_score(train, pt).cpu().numpy().astype(np.float64)
    th, eh = train.cpu().numpy(), test.cpu().numpy()
    ref = th.astype(np.float64) @ oracle_mod.fim_solve(oracle_mod.fim(th)[0], lam, eh.astype(np.float64)).T
    cond = np.linalg.cond(oracle_mod.fim(th)[0] + lam * np.eye(k))
    scale = np.linalg.norm(ref, axis=0, keepdims=True) / np.sqrt(n)
    assert (np.abs(sc - ref) / scale).max() <= 64 * cond * 2.0 ** -23


# Sizes at which the one-launch kernels change shape: one block, one block and a row, a last block of one row; the first
# trailing update just within / beyond one thread block per tile (k = 1,088 / 1,152); row strides that rule out 16-byte loads.
@pytest.mark.parametrize("k,M,pad", [(1, 1, 0), (63, 2, 1), (64, 40, 0), (65, 5, 3), (128, 600, 4), (129, 33, 1), (320, 1, 0),
                                     (576, 130, 2), (1088, 260, 0), (1152, 300, 1), (1345, 37, 4), (256, 5000, 0)])
def test_factor_and_apply_shapes(G, k, M, pad):
    n = 2 * k + 3
    X = _compressed(n, k, 40 + k)
    wide = torch.full((k, k + pad), float("nan"), device="cuda")
    F = wide[:, :k]
    G.grass_fim(X, out=F)
    A = torch.tril(F).double()
    A = A + torch.tril(A, -1).T + 0.05 * torch.eye(k, device="cuda", dtype=torch.float64)
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    G.grass_fim_factor(F, 0.05, dev_status=st)
    wide_b = torch.full((M, k + pad), float("nan"), device="cuda")
    Bm = wide_b[:, :k]
    Bm.copy_(_compressed(M, k, 41 + k))
    b = Bm.double()
    G.grass_fim_apply(F, Bm)
    assert int(st.item()) == 0
    assert pad == 0 or (torch.isnan(wide[:, k:]).all() and torch.isnan(wide_b[:, k:]).all())
    # backward error of a factorisation and two substitutions with k-term fp32 sums: rounding errors of independent
    # sign add like sqrt(k) 2^-24, three passes, two standard deviations
    u = 6.0 * k ** 0.5 * 2.0 ** -24
    L = torch.tril(F).double()
    assert (L @ L.T - A).norm() <= u * A.norm()
    x = Bm.double()
    assert (x @ A - b).norm() <= u * A.norm() * x.norm()


# Many right-hand sides are solved block column by block column: ragged last block, ragged last tile of rows, row strides
@pytest.mark.parametrize("k,M,pad", [(63, 16_400, 1), (64, 16_400, 0), (130, 16_411, 3), (513, 16_411, 2), (1_030, 5_003, 0)])
def test_apply_many_right_hand_sides(G, k, M, pad):
    X = _compressed(2 * k + 3, k, 70 + k)
    F = torch.full((k, k + pad), float("nan"), device="cuda")[:, :k]
    G.grass_fim(X, out=F)
    A = F.double() + 0.05 * torch.eye(k, device="cuda", dtype=torch.float64)
    G.grass_fim_factor(F, 0.05)
    wide = torch.full((M, k + pad), float("nan"), device="cuda")
    Bm = wide[:, :k]
    Bm.copy_(_compressed(M, k, 71 + k))
    b, few = Bm.double(), Bm[:100].clone()
    G.grass_fim_apply(F, Bm)
    assert pad == 0 or torch.isnan(wide[:, k:]).all()
    x, y = Bm.double(), G.grass_fim_apply(F, few).double()
    # the bound of test_factor_and_apply_shapes, and the same for the difference from a solve of the first rows alone
    u = 6.0 * k ** 0.5 * 2.0 ** -24
    assert (x @ A - b).norm() <= u * A.norm() * x.norm()
    assert ((x[:100] - y) @ A).norm() <= 2.0 * u * A.norm() * y.norm()


# Pivots at both ends of the fp32 range: below 2^-126 they are subnormal, above 2^126 their reciprocals are
@pytest.mark.parametrize("scale", [1.0e-38, 1.0, 1.2e38])
def test_factor_of_scaled_matrices(G, scale):
    k = 200
    X = _compressed(4 * k, k, 5)
    C = torch.corrcoef(X.double().T)
    A = ((0.3 * C + 0.7 * torch.eye(k, device="cuda", dtype=torch.float64)) * scale).float()
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    L = torch.tril(G.grass_fim_factor(A.clone(), 0.0, dev_status=st)).double() / scale ** 0.5
    assert int(st.item()) == 0
    # the bound of test_factor_and_apply_shapes for one pass; a subnormal matrix is updated in steps of 2^-149, one update
    # for every 8 columns
    A = A.double() / scale
    assert (L @ L.T - A).norm() <= 2.0 * k ** 0.5 * 2.0 ** -24 * A.norm() + (k / 8) * k * 2.0 ** -149 / scale


# The roots and reciprocals of the pivots themselves, as the factors of 2 x 2 blocks [d x; x y] show them: sqrt(d), x / sqrt(d) and
# sqrt(y - x^2 / d), here with x = d and y = 2 d, over all of fp32 that leaves room for them.
def test_roots_and_reciprocals_of_pivots(G):
    k = 4096
    gen = torch.Generator(device="cuda").manual_seed(3)
    d = torch.exp2(torch.rand(k // 2, generator=gen, device="cuda") * 251.0 - 125.0)
    at = torch.arange(0, k, 2, device="cuda")
    A = torch.zeros((k, k), device="cuda")
    A[at, at], A[at + 1, at], A[at, at + 1], A[at + 1, at + 1] = d, d, d, 2 * d
    L = G.grass_fim_factor(A, 0.0).double()
    u, root = 2.0 ** -24, d.double().sqrt()
    # against CUDA's square root, which is correctly rounded: an ulp and a half
    assert ((L[at, at] - torch.sqrt(d).double()).abs() <= 3.0 * u * root).all()
    # x times the reciprocal root: its error and one rounding
    assert ((L[at + 1, at] - root).abs() <= 4.0 * u * root).all()
    # the second pivot is 2 d - d (d / d): a reciprocal one ulp off (2 u) and two roundings, half of it after the root
    assert ((L[at + 1, at + 1] - root).abs() <= (3.0 + 2.0) * u * root).all()
    # subnormal pivots have roots like any other
    s = torch.rand(4096, generator=gen, device="cuda") * 2.0 ** -126 + 2.0 ** -127
    A = torch.diag(s)
    L = torch.diagonal(G.grass_fim_factor(A, 0.0)).double()
    assert ((L - s.double().sqrt()).abs() <= 3.0 * u * s.double().sqrt()).all()


# one sample, fewer samples than a step, a chunk boundary at 8,192; tiles on the diagonal alone, a ragged second tile, many
# tiles (pairs instead of clusters of eight); columns that start off a 16-byte boundary
@pytest.mark.parametrize("n,k,off", [(1, 128, 0), (31, 129, 0), (33, 127, 1), (8_192, 64, 0), (8_200, 200, 3), (700, 900, 0)])
def test_fim_shapes(G, n, k, off):
    X = _compressed(n, k + off + 3, 60 + k)[:, off:off + k]
    F = G.grass_fim(X).double()
    Xd = X.double()
    ref, absum = Xd.T @ Xd / n, Xd.abs().T @ Xd.abs() / n
    # six bf16 products keep each product to 2^-23; accumulators are truncated once per 16 samples
    assert ((F - ref).abs() <= 2.0 ** -22 * absum + 2.0 * (n / 16 + 64) ** 0.5 * 2.0 ** -23 * absum).all()
    assert (F - F.T).abs().max() <= 2.0 ** -21 * absum.max()


# A wait that expires in one thread block of a cluster spoils what the others go on with: all rows of all clusters are NaN, whichever
# block it was, and the next call is sound.  (The block takes its waits as expired without having waited, and then waits.)
@pytest.mark.parametrize("k,M,block", [(1_030, 40, 0), (1_030, 40, 5), (300, 33, 2), (130, 700, 1)])
def test_expired_wait_leaves_no_finite_row(G, tune, k, M, block):
    F = G.grass_fim(_compressed(k + 64, k, 80 + k))
    G.grass_fim_factor(F, 0.1)
    B = _compressed(M, k, 81 + k)
    ref = G.grass_fim_apply(F, B.clone())
    tune(fim_expire=block)
    got = G.grass_fim_apply(F, B.clone())
    tune(fim_expire=None)
    assert torch.isnan(got).all()
    assert torch.equal(G.grass_fim_apply(F, B.clone()), ref)


# Every number of right-hand sides per cluster with every number of thread blocks, whichever the sizes would choose: as many blocks
# of 64 columns as thread blocks and one more (the buffers of the solved blocks come round), the last one ragged or whole, and
# several rounds; rows that leave one over, a last cluster of one row; strides that rule out 16-byte copies.
@pytest.mark.parametrize("rows", [2, 4, 8, 16, 32])
@pytest.mark.parametrize("blocks", [1, 2, 4, 8])
def test_apply_every_cluster_shape(G, tune, blocks, rows):
    for k, M, pad in ((64 * blocks, 2 * rows + 1, 0), (64 * blocks + 1, rows, 1), (64 * (2 * blocks + 1) + 37, 3 * rows - 1, 3),
                      (64 * (3 * blocks + 2), rows + 1, 4)):
        X = _compressed(2 * k + 3, k, 90 + k)
        F = torch.full((k, k + pad), float("nan"), device="cuda")[:, :k]
        G.grass_fim(X, out=F)
        A = F.double() + 0.05 * torch.eye(k, device="cuda", dtype=torch.float64)
        G.grass_fim_factor(F, 0.05)
        wide = torch.full((M + 1, k + pad), float("nan"), device="cuda")
        Bm = wide[:M, :k]
        Bm.copy_(_compressed(M, k, 91 + k))
        b = Bm.double()
        tune(fim_rows=rows, fim_cluster=blocks)
        G.grass_fim_apply(F, Bm)
        assert torch.isnan(wide[M]).all() and (pad == 0 or torch.isnan(wide[:, k:]).all())
        x = Bm.double()
        # the bound of test_factor_and_apply_shapes
        u = 6.0 * k ** 0.5 * 2.0 ** -24
        assert (x @ A - b).norm() <= u * A.norm() * x.norm(), (k, M)
        # row by row, so that no row hides behind the others
        assert ((x @ A - b).norm(dim=1) <= 4.0 * u * A.norm() * x.norm(dim=1)).all(), (k, M)


# The block columns' path takes few right-hand sides as well: one row, a last tile of one row, a ragged last block
@pytest.mark.parametrize("k,M,pad", [(1, 1, 0), (64, 65, 0), (130, 1, 3), (193, 129, 1)])
def test_apply_block_columns_of_few_rows(G, tune, k, M, pad):
    F = torch.full((k, k + pad), float("nan"), device="cuda")[:, :k]
    G.grass_fim(_compressed(2 * k + 3, k, 97 + k), out=F)
    A = F.double() + 0.05 * torch.eye(k, device="cuda", dtype=torch.float64)
    G.grass_fim_factor(F, 0.05)
    B = _compressed(M, k, 98 + k)
    tune(fim_cluster=0)
    x = G.grass_fim_apply(F, B.clone()).double()
    u = 6.0 * k ** 0.5 * 2.0 ** -24
    assert (x @ A - B.double()).norm() <= u * A.norm() * x.norm()


# ... and the sizes' own choice where it is one of the larger shapes (32 rows in one block and in two, 16 in eight)
@pytest.mark.parametrize("k,M", [(64, 2_500), (1_216, 1_200), (1_792, 1_750), (1_280, 140), (512, 8), (500, 2_900)])
def test_apply_sizes_of_the_larger_shapes(G, k, M):
    F = G.grass_fim(_compressed(2 * k + 3, k, 95 + k))
    A = F.double() + 0.05 * torch.eye(k, device="cuda", dtype=torch.float64)
    G.grass_fim_factor(F, 0.05)
    B = _compressed(M, k, 96 + k)
    x = G.grass_fim_apply(F, B.clone()).double()
    u = 6.0 * k ** 0.5 * 2.0 ** -24
    assert (x @ A - B.double()).norm() <= u * A.norm() * x.norm()
