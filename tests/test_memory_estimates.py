"""What a solve is counted with and how it is split do not depend on each other.

Pass 1 may take more row splits than its memory is counted with (their partial sums stay within
the working set's allowance): estimates, what set_data takes and what a server admits are those of
the counted splits, and the splits, hence the bits and what a checkpoint continues to, are the same
whatever memory there is.
"""
import os
import shutil

import numpy as np
import pytest

# 24 feature tiles by 2 row blocks: 7 row splits make two waves of CTAs on 148 to 152 SMs; 9 fill them
CASE = dict(loss="hinge", reg="l2", lam=1e-4, sigma=6.0, rho=1.0, D=3000, R=2, C=3, seed=5, m=1, prec="split_bf16")
N, DIM, COUNTED = 20_011, 33, 7


@pytest.fixture(scope="module")
def rff():
    if not shutil.which("nvcc") and not os.path.exists("/usr/local/cuda/bin/nvcc"):
        pytest.skip("nvcc not available")
    import __graft_entry__
    __graft_entry__.build()
    import paper_1409_0940_gb300
    return paper_1409_0940_gb300


def estimate(rff, monkeypatch, splits=None):
    if splits:
        monkeypatch.setenv("RFF_PASS1_SPLITS", str(splits))
    else:
        monkeypatch.delenv("RFF_PASS1_SPLITS", raising=False)
    got = rff.rff_admm_estimate_bytes(rff.make_params(**CASE), N, DIM)
    monkeypatch.delenv("RFF_PASS1_SPLITS", raising=False)
    return got


def test_estimates_count_the_fewest_splits(rff, monkeypatch):
    assert estimate(rff, monkeypatch) == estimate(rff, monkeypatch, COUNTED)
    assert estimate(rff, monkeypatch)[0] < estimate(rff, monkeypatch, 9)[0]


def test_estimates_count_features_not_tiles(rff):
    """Rows padded for the kernels' 16-byte copies come out of the allowance."""
    def fp32(D, C, n):
        return rff.rff_admm_estimate_bytes(rff.make_params(prec="fp32", D=D, R=1, C=C, m=1), n, 10)
    # the set-up's chunk of Z: 32,768 rows of D floats (the factorisation's scratch is the same for both)
    (r1, p1), (r2, p2) = fp32(129, 1, 40_000), fp32(160, 1, 40_000)
    assert (p2 - r2) - (p1 - r1) == 32_768 * 31 * 4 + 16 * (160 ** 2 - 129 ** 2)
    # the factors (the slots are the same for both)
    assert fp32(8 * 132, 8, 4000)[0] - fp32(8 * 129, 8, 4000)[0] == 4 * 8 * (132 ** 2 - 129 ** 2)


def train(rff, data, limit=0, iters=6, state=None):
    s = rff.Solver(**CASE)
    if limit:
        rff.rff_admm_set_memory_limit(s.h, limit)
    s.set_data(*data)
    if state is not None:
        s.set_state(state)
    s.solve(iters, stats=False)
    return s


@pytest.mark.gpu
def test_bits_do_not_depend_on_the_memory_there_is(rff, monkeypatch):
    import synth
    data = synth.binary(n=N, d=DIM, seed=2)
    free = train(rff, data, iters=3)
    assert free.profile()["nsplit"] > COUNTED
    state = free.get_state()
    free.solve(3, stats=False)
    # the least that set_data takes: the counted peak without the staging of the inputs
    slots = 2 * (-(-(-(-N // 2)) // 128) * 128)
    least = estimate(rff, monkeypatch, COUNTED)[1] - N * (DIM + 1) * 4 - slots * 64 * 4
    tight = train(rff, data, limit=least)
    assert np.array_equal(tight.weights(), free.weights())
    resumed = train(rff, data, limit=least, iters=3, state=state)
    assert np.array_equal(resumed.weights(), free.weights())
    with pytest.raises(rff.RffError) as e:
        train(rff, data, limit=least - 1)
    assert e.value.status == rff.RFF_ENOMEM
    for s in (free, tight, resumed):
        s.close()


@pytest.mark.gpu
def test_a_server_admits_the_counted_peak(rff, monkeypatch):
    import synth
    X, Y = synth.binary(n=N, d=DIM, seed=2)
    alone = train(rff, (X, Y))
    srv = rff.rff_server_create(estimate(rff, monkeypatch, COUNTED)[1], 1)
    rid = rff.rff_server_submit_solve(srv, rff.make_params(**CASE), X, Y, 6)
    done = []
    for _ in range(300):
        done = rff.rff_server_poll(srv, 4, 1000)
        if done:
            break
    assert [c["status"] for c in done] == [rff.RFF_OK]
    W = rff.rff_server_get_weights(srv, rid, np.empty((CASE["D"], 1), np.float32))
    assert np.array_equal(W, alone.weights())
    rff.rff_server_destroy(srv)
    alone.close()
