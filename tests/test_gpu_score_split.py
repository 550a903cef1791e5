"""Scoring of small batches, which the tensor-core path splits over the feature groups.

The groups' sums are added in one order whether one CTA takes them all or several share them, so
a row's scores are the same bits in any batch; against the float64 features they stay within the
split path's tolerance.  Sizes: one row, one less and one more than a 128-row tile, a whole wave
of the SMs plus a remainder; one feature group, three (the last of them short), and thirteen.
"""
import numpy as np
import pytest

from oracle import rff as orff

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rff():
    import paper_1409_0940_gb300 as m
    return m


@pytest.mark.parametrize("prec", ["split_bf16", "cached_z"])
@pytest.mark.parametrize("D,C", [(100, 1), (2500, 2), (13000, 3)])
def test_scores_do_not_depend_on_the_batch(rff, prec, D, C):
    rng = np.random.default_rng(3)
    d, m, n = 21, 3, 400
    X = rng.standard_normal((n, d)).astype(np.float32)
    Y = np.sign(rng.standard_normal((n, m))).astype(np.float32)
    s = rff.Solver(loss="squared", reg="l2", lam=1e-3, sigma=4.0, rho=1.0, D=D, R=1, C=C, seed=9, m=m, prec=prec)
    s.set_data(X, Y)
    s.solve(2)
    W = s.weights()
    Q = rng.standard_normal((160 * 128 + 45, d)).astype(np.float32)
    full = s.predict(Q)
    for q in (1, 127, 129, 1000, 152 * 128 + 1):
        assert np.array_equal(s.predict(np.ascontiguousarray(Q[:q])), full[:q])
    rows = np.r_[0:50, Q.shape[0] - 50:Q.shape[0]]
    ref = orff.features_block(Q[rows], 9, 4.0, D, 0, D) @ W.astype(np.float64)
    assert np.linalg.norm(full[rows] - ref) <= 1e-4 * np.linalg.norm(ref)
    s.close()


# sums below the smallest normal FP32 number keep their value whichever way they are added: targets
# of 1e-36 and 1e-38 train weights, and give group sums, that are mostly subnormal
@pytest.mark.parametrize("prec", ["split_bf16", "cached_z"])
@pytest.mark.parametrize("scale", [1e-36, 1e-38])
def test_tiny_scores_do_not_depend_on_the_batch(rff, prec, scale):
    rng = np.random.default_rng(3)
    X = rng.standard_normal((400, 21)).astype(np.float32)
    Y = (np.sign(rng.standard_normal((400, 3))) * scale).astype(np.float32)
    s = rff.Solver(loss="squared", reg="l2", lam=1e-3, sigma=4.0, rho=1.0, D=13000, R=1, C=3, seed=9, m=3, prec=prec)
    s.set_data(X, Y)
    s.solve(2)
    W = s.weights()
    Q = rng.standard_normal((160 * 128 + 45, 21)).astype(np.float32)
    full = s.predict(Q)
    for q in (1, 1000):
        assert np.array_equal(s.predict(np.ascontiguousarray(Q[:q])), full[:q])
    # The weights' FP16 split is scaled by at most 2^108, so a weight is off by up to 2^-133 (uniformly:
    # 2^-133 / sqrt 3 in the root mean square), and a score, with D features of square sum about 1, by
    # as much; four times that, beside the split path's 1e-4
    ref = orff.features_block(Q[:50], 9, 4.0, 13000, 0, 13000) @ W.astype(np.float64)
    split = 4 * np.sqrt(ref.size / 3.0) * 2.0 ** -133
    assert np.linalg.norm(full[:50].astype(np.float64) - ref) <= 1e-4 * np.linalg.norm(ref) + split
    s.close()


# refused queries leave the caller's scores alone, on the device (where the copy out looks at the
# check's outcome itself) and on the host
@pytest.mark.parametrize("prec,fmap", [("split_bf16", "fourier"), ("fp32", "laplace"), ("cached_z", "tensorsketch")])
@pytest.mark.parametrize("where", ["device", "host"])
def test_refused_queries_leave_the_scores_alone(rff, prec, fmap, where):
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(3)
    X = rng.random((300, 7)).astype(np.float32)
    Y = np.sign(rng.standard_normal((300, 2))).astype(np.float32)
    s = rff.Solver(loss="squared", lam=1e-3, sigma=2.0, D=200, R=1, C=2, seed=9, m=2, prec=prec, feature_map=fmap)
    s.set_data(X, Y)
    s.solve(2)
    good = rng.random((200, 7)).astype(np.float32)
    want = s.predict(good)
    bad = {"nan": np.nan}
    if prec == "split_bf16":
        bad["range"] = 1e30      # beyond the FP16 split's range
    if fmap == "laplace":
        bad["negative"] = -1.0

    def call(Q):
        out = np.full((200, 2), 7.0, np.float32)
        if where == "host":
            return out, lambda: s.predict(Q, out), lambda: out
        q, o = torch.from_numpy(Q).cuda(), torch.from_numpy(out).cuda()
        return out, lambda: s.predict(q, o), lambda: o.cpu().numpy()

    for value in bad.values():
        Q = good.copy()
        Q[150, 3] = value
        before, run, after = call(Q)
        with pytest.raises(rff.RffError) as e:
            run()
        assert e.value.status == rff.RFF_EINVAL
        assert np.array_equal(after(), np.full((200, 2), 7.0, np.float32))
    _, run, after = call(good)
    run()
    assert np.array_equal(after(), want)
    s.close()
