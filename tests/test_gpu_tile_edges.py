"""Edges of the FP32 tiles, the set-up's batches and the splits of work over CTAs.

Where work is split (feature parts over a cluster's CTAs, K chunks of a factor product, the
factorisation beside the forward sweep, row blocks of the outer form) the sums keep their order or
their float-float accuracy: results are the same bits where the order is the same, and within the
FP32 path's tolerance of the float64 oracle everywhere.
"""
import numpy as np
import pytest

from oracle import admm, rff as orff

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rff():
    import paper_1409_0940_gb300 as m
    return m


def data(n, d, m, seed=3):
    rng = np.random.default_rng(seed)
    X = rng.standard_normal((n, d)).astype(np.float32)
    Y = np.sign(rng.standard_normal((n, m))).astype(np.float32)
    return X, Y


def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


# 1, 3, 6 and 20 feature tiles (none, clusters of 4 and 8); d below, at and past a K stage; one to
# sixteen 16-column runs, the parked and the float-float sums, every number of M rows per stage
@pytest.mark.parametrize("D,C,d,m", [(100, 1, 1, 1), (300, 2, 32, 20), (700, 1, 33, 70), (2500, 3, 66, 150),
                                     (300, 1, 5, 256)])
def test_fp32_scores_do_not_depend_on_the_batch(rff, D, C, d, m):
    X, Y = data(300, d, m)
    s = rff.Solver(loss="squared", reg="l2", lam=1e-3, sigma=4.0, rho=1.0, D=D, R=1, C=C, seed=9, m=m, prec="fp32")
    s.set_data(X, Y)
    s.solve(2)
    W = s.weights()
    Q = np.random.default_rng(5).standard_normal((155 * 128 + 45, d)).astype(np.float32)
    full = s.predict(Q)
    for q in (1, 127, 129, 1000, 152 * 128 + 1):
        assert np.array_equal(s.predict(np.ascontiguousarray(Q[:q])), full[:q])
    rows = np.r_[0:40, Q.shape[0] - 40:Q.shape[0]]
    ref = orff.features_block(Q[rows], 9, 4.0, D, 0, D) @ W.astype(np.float64)
    # FP32 sums of D products of magnitude |z| |w|: the path's 1e-5
    assert rel(full[rows], ref) <= 1e-5
    s.close()


# passes, factor products and Gram matrices on ragged blocks: a Gram form with one short tile and
# K = 87 (the tail of a 32-K chunk), one with m = 150 (parked factor sums), one whose factor
# products go to clusters, and outer forms (fewer rows than features) of 5 and 7 uneven row blocks
@pytest.mark.parametrize("prec,tol", [("fp32", 1e-5), ("split_bf16", 1e-4)])
@pytest.mark.parametrize("n,d,m,D,R,C", [(1003, 17, 1, 87, 1, 1), (1003, 5, 150, 261, 2, 2), (700, 9, 3, 600, 1, 1),
                                         (651, 40, 2, 1200, 5, 3), (903, 12, 20, 300, 7, 1)])
def test_ragged_solves_match_the_oracle(rff, prec, tol, n, d, m, D, R, C):
    X, Y = data(n, d, m, seed=n)
    kw = dict(loss="squared", reg="l2", lam=1e-3, sigma=4.0, rho=1.0, D=D, R=R, C=C, seed=5)
    ref = admm.admm(admm.Problem(X, Y, **kw), 8)["Wbar"]
    s = rff.Solver(prec=prec, m=m, **kw)
    s.set_data(X, Y)
    s.solve(8, stats=False)
    assert rel(s.weights(), ref) <= tol
    s.close()


# With a memory limit the forward sweep runs after the factorisation instead of beside it, and a
# TensorSketch solve forms its features in row chunks (9,000 rows of 8,192 features: 256 MB take 8,192
# rows) instead of whole
@pytest.mark.parametrize("kw,d,n", [
    (dict(D=900, R=2, C=3, prec="split_bf16"), 10, 2000),
    (dict(D=900, R=2, C=1, prec="fp32"), 10, 2000),
    (dict(D=2000, R=6, C=2, prec="fp32"), 10, 1500),
    (dict(D=8192, R=1, C=2, prec="cached_z", feature_map="tensorsketch", degree=2, coef0=1.0), 20, 9000)])
def test_a_memory_limit_changes_no_result(rff, kw, d, n):
    X, Y = data(n, d, 4)
    got = []
    for limit in (0, 4 << 30):
        s = rff.Solver(loss="hinge", reg="l2", lam=1e-4, sigma=4.0, rho=1.0, seed=5, m=4, **kw)
        if limit:
            rff.rff_admm_set_memory_limit(s.h, limit)
        s.set_data(X, Y)
        s.solve(4, stats=False)
        got.append(s.weights())
        s.close()
    assert np.array_equal(got[0], got[1])


# The outer form's set-up takes Z^T of several row blocks at once and factors blocks in batches.  Of
# 100 row blocks by 2 column blocks, limits of some MB above the resident set leave room for batches
# of 1 block, of 31 (that begin and end within a row of the grid) and of 133, whose row blocks are more
# than the 46 that Z^T is then formed for at once
@pytest.mark.parametrize("prec,tol", [("fp32", 1e-5), ("split_bf16", 1e-4)])
def test_outer_set_up_in_batches(rff, prec, tol):
    kw = dict(loss="squared", reg="l2", lam=1e-3, sigma=4.0, rho=1.0, D=4201, R=100, C=2, seed=5)
    X, Y = data(12_737, 6, 2)
    ref = admm.admm(admm.Problem(X, Y, **kw), 4)["Wbar"]
    resident = rff.rff_admm_estimate_bytes(rff.make_params(prec=prec, m=2, **kw), *X.shape)[0]
    got = []
    for extra in (0, 290, 310, 370):
        s = rff.Solver(prec=prec, m=2, **kw)
        if extra:
            rff.rff_admm_set_memory_limit(s.h, resident + (extra << 20))
        s.set_data(X, Y)
        s.solve(4, stats=False)
        got.append(s.weights())
        s.close()
    assert rel(got[0], ref) <= tol
    assert all(np.array_equal(g, got[0]) for g in got)


# ... and, without a limit, more row blocks than 256 MB of Z^T hold (36 of 40)
def test_outer_set_up_of_more_row_blocks_than_fit_at_once(rff):
    kw = dict(loss="squared", reg="l2", lam=1e-3, sigma=4.0, rho=1.0, D=2100, R=40, C=1, seed=5)
    X, Y = data(33_501, 6, 2)
    ref = admm.admm(admm.Problem(X, Y, **kw), 3)["Wbar"]
    s = rff.Solver(prec="fp32", m=2, **kw)
    s.set_data(X, Y)
    s.solve(3, stats=False)
    assert rel(s.weights(), ref) <= 1e-5
    s.close()


# the row losses by outputs per lane: 2, 3, 5 (of 4) and 8 (of 7), with ragged lanes; their step tests
# go through another kernel
@pytest.mark.parametrize("loss", ["multinomial", "crammer_singer"])
@pytest.mark.parametrize("m", [40, 70, 115, 200])
def test_row_losses_by_outputs_per_lane(rff, loss, m):
    rng = np.random.default_rng(m)
    X = rng.standard_normal((700, 9)).astype(np.float32)
    Y = np.full((700, m), -1.0, np.float32)
    Y[np.arange(700), rng.integers(0, m, 700)] = 1.0
    kw = dict(loss=loss, reg="l2", lam=1e-3, sigma=3.0, rho=1.0, D=300, R=2, C=2, seed=5)
    ref = admm.admm(admm.Problem(X, Y, **kw), 8)["Wbar"]
    for prec, tol in (("fp32", 1e-5), ("split_bf16", 1e-4)):
        s = rff.Solver(prec=prec, m=m, **kw)
        s.set_data(X, Y)
        s.solve(8, stats=False)
        assert rel(s.weights(), ref) <= tol, prec
        s.close()


# the diagonal blocks multiply by 1 / pivot: pivots whose reciprocal or square is out of range factor
# as any other (20 copies of one 3 x 3 block with an exact factor; one subnormal pivot among ones)
@pytest.mark.parametrize("e", [-1060, -1000, -100, 0, 100, 1000, 1018])
def test_cholesky_of_tiny_and_huge_pivots(rff, e):
    torch = pytest.importorskip("torch")
    T = np.array([[2.0, 0, 0], [1, 2, 0], [0, 1, 4]])
    L = np.kron(np.eye(20), T) * 2.0 ** (e // 2)
    A = np.kron(np.eye(20), T @ T.T) * 2.0 ** (e - e // 2) * 2.0 ** (e // 2)
    if e == -1060:
        L[3:6, 3:6], A[3:6, 3:6] = np.diag([1.0, 2.0 ** -525, 1.0]), np.diag([1.0, 2.0 ** -525 * 2.0 ** -525, 1.0])
    At, info = torch.from_numpy(A[None].copy()).cuda(), torch.zeros(1, dtype=torch.int32, device="cuda")
    rff.rff_cholesky_f64(At, info)
    assert info.item() == 0
    assert np.array_equal(At[0].cpu().numpy(), L)


@pytest.mark.parametrize("nf", [1, 127, 129, 1000])
@pytest.mark.parametrize("d", [1, 33, 70])
def test_features_do_not_depend_on_the_number_of_rows(rff, d, nf):
    """Few tiles go one to a block of threads, many two to one: every row has the same bits either way."""
    import torch
    n, few = 20100, 130   # 158 row tiles: pairs on any GPU of up to 157 SMs; 2 x 8 tiles: singles
    g = torch.Generator(device="cuda").manual_seed(d)
    X = torch.randn(n, d, device="cuda", generator=g)
    full, part = torch.empty(n, nf, device="cuda"), torch.empty(few, nf, device="cuda")
    rff.rff_features(X, 7, 1.5, nf, 0, nf, "fp32", full)
    for lo in (0, n - few):
        rff.rff_features(X[lo:lo + few].contiguous(), 7, 1.5, nf, 0, nf, "fp32", part)
        assert torch.equal(part, full[lo:lo + few])
    want = orff.features_block(X[n - few:].cpu().numpy(), 7, 1.5, nf, 0, nf)
    # float32 dot products of length d and the float32 cosine (as the features against the oracle elsewhere)
    assert np.abs(part.cpu().numpy() - want).max() < 1e-5 * max(1.0, np.sqrt(d / 16)) * np.sqrt(2.0 / nf)
