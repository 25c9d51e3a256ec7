"""C-first sweeps that only read R (a pass serves several k), beyond the SMs'
shared memory: each count of vectors a thread holds, K that is and is not a multiple
of a pass's k, columns that leave part of a chunk, of a round of the groups
and of a unit.  Against the FP64 oracle's Algorithm 2 and the kernel that writes R.
"""

import numpy as np
import pytest

from oracle import did_oracle as O
from synth import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def did():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1802_08938_gb300 as did
    return did


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a, np.float64) - b) / np.linalg.norm(b))


def run(did, X, B0, C0, sweeps, **kw):
    M, N = X.shape
    with did.Context(np.ascontiguousarray(X.T), M, N, B0.shape[1], B_init=np.ascontiguousarray(B0.T), C_init=C0,
                     order=did.DID_ORDER_DID, **kw) as ctx:
        ctx.sweep(sweeps)
        B, C = ctx.factors()
        return dict(B=B, C=C, R=ctx.residual(), trace=ctx.trace(), f=ctx.objective(), info=ctx.info())


SHAPES = [(64, 150001, 7), (130, 70003, 4), (784, 12001, 5), (1030, 9001, 1), (2064, 4503, 9), (5003, 1999, 3),
          (9000, 1051, 6), (12000, 801, 3), (600, 16001, 66), (520, 20011, 128)]


@pytest.mark.parametrize("M,N,K", SHAPES)
def test_float32_matches_oracle(did, M, N, K):
    X, _, _ = W.planted(M, N, K, seed=M + N, sigma=0.05)
    B0, C0 = W.init_factors(M, N, K, 5)
    ref = O.factor(X, B0, C0, order="dbcd", max_iter=3, stop="none")
    got = run(did, X, B0, C0, 3)
    rows = 4 * got["info"]["vecs_per_thread"]
    assert got["info"]["sweep_form"] == did.DID_FORM_READ_ONLY
    assert got["info"]["pass_blocks"] == (4 if rows <= 16 else 2)
    again = run(did, X, B0, C0, 3)
    eager = run(did, X, B0, C0, 3, flags=did.DID_FLAG_EAGER_WRITEBACK)
    eB, eC = rel(got["B"], ref["B"]), rel(got["C"], ref["C"])
    eF = float(np.max(np.abs(got["trace"] - ref["trace"]) / ref["trace"]))
    print("C-first read-only M=%d N=%d K=%d: relB %.3g relC %.3g relf %.3g (eager %.3g %.3g)" % (
        M, N, K, eB, eC, eF, rel(eager["B"], ref["B"]), rel(eager["C"], ref["C"])))
    # float32 dots over up to 150001 terms and the refresh's 2^-21 |B||C|: a few 1e-7 each, 1e-5 with margin
    assert eB <= 1e-5 and eC <= 1e-5 and eF <= 1e-5
    assert np.array_equal(got["B"], again["B"]) and np.array_equal(got["C"], again["C"])
    assert np.array_equal(got["trace"], again["trace"])
    Rd = X.astype(np.float64) - got["B"].astype(np.float64) @ got["C"].astype(np.float64)
    S = np.abs(got["B"]).astype(np.float64) @ got["C"].astype(np.float64)
    assert np.all(np.abs(got["R"] - Rd) <= 2.0 ** -17 * S + 2.0 ** -22 * np.abs(Rd) + 1e-6)


@pytest.mark.parametrize("M,N,K", [(130, 70003, 7), (784, 24001, 20), (2064, 9003, 9), (9000, 2051, 30)])
def test_bfloat16_residual(did, M, N, K):
    X, _, _ = W.planted(M, N, K, seed=M + N, sigma=0.05)
    B0, C0 = W.init_factors(M, N, K, 5)
    ref = O.factor(X, B0, C0, order="dbcd", max_iter=3, stop="none")
    got = run(did, X, B0, C0, 3, precision=did.DID_BF16R, refresh_every=2)
    assert got["info"]["sweep_form"] == did.DID_FORM_READ_ONLY
    assert got["info"]["refreshes"] == 1
    eB, eC = rel(got["B"], ref["B"]), rel(got["C"], ref["C"])
    print("C-first read-only bfloat16 M=%d N=%d K=%d: relB %.3g relC %.3g" % (M, N, K, eB, eC))
    # R is rounded by up to 2^-9 of an entry once a sweep; a contraction carries at most that share of |R| |b|
    assert eB <= 3 * 2.0 ** -9 and eC <= 3 * 2.0 ** -9
    assert abs(got["f"] - ref["trace"][-1]) <= 1e-3 * ref["trace"][-1]


def test_stopping_and_zero_norms(did):
    M, N, K = 800, 12003, 4
    X, _, _ = W.planted(M, N, K, seed=1, sigma=0.05)
    B0, C0 = W.init_factors(M, N, K, 2)
    B0[:, 2] = 0.0                      # ||b_3|| = 0: c_3 is left unchanged until b_3 is updated
    ref = O.factor(X, B0, C0, order="dbcd", max_iter=60, tol=1e-2, stop="relchange")
    with did.Context(np.ascontiguousarray(X.T), M, N, K, B_init=np.ascontiguousarray(B0.T), C_init=C0,
                     order=did.DID_ORDER_DID) as ctx:
        iters, f = ctx.factor(60, 1e-2)
        B, C = ctx.factors()
        assert iters == ref["iters"] and ctx.info()["degenerate_events"] >= 1
    assert rel(B, ref["B"]) <= 1e-5 and rel(C, ref["C"]) <= 1e-5


def test_expired_wait_is_reported(did):
    M, N, K = 800, 12003, 3
    X, _, _ = W.planted(M, N, K, seed=1, sigma=0.05)
    with did.Context(np.ascontiguousarray(X.T), M, N, K, seed=0, timeout_ns=10 ** 7, debug_barrier_extra=1,
                     order=did.DID_ORDER_DID) as ctx:
        with pytest.raises(did.DIDError) as e:
            ctx.sweep(1)
        assert e.value.status == did.DID_ETIMEOUT
        B, C = ctx.factors()
        assert np.isfinite(B).all() and (B >= 0).all() and np.isfinite(C).all() and (C >= 0).all()


def test_expired_wait_ends_the_queued_sweeps(did):
    """After an expired wait the sweeps queued behind it change nothing: B and C
    are those that one sweep leaves, whatever the number asked for, and the
    context goes on from them."""
    M, N, K = 800, 12003, 3
    X, _, _ = W.planted(M, N, K, seed=1, sigma=0.05)
    left = []
    for n in (1, 6, 6):
        with did.Context(np.ascontiguousarray(X.T), M, N, K, seed=0, timeout_ns=10 ** 7, debug_barrier_extra=1, order=did.DID_ORDER_DID) as ctx:
            with pytest.raises(did.DIDError) as e:
                ctx.sweep(n)
            assert e.value.status == did.DID_ETIMEOUT
            left.append((*ctx.factors(), ctx.trace(), ctx.info()["sweeps_done"]))
    for B, C, trace, done in left[1:]:
        assert np.array_equal(B, left[0][0]) and np.array_equal(C, left[0][1])
        assert len(trace) == 1 and done == 0
