"""Sweeps of a residual that stays in the SMs' shared memory, the CTAs
exchanging flagged words: both orders, both precisions, one CTA to all of
them, slices of one row and of many, one column a CTA and many, K = 1, and
launches of one sweep and of several.  Against the FP64 oracle.
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
                     **kw) as ctx:
        assert ctx.info()["sweep_form"] == did.DID_FORM_RESIDENT
        for n in sweeps:
            ctx.sweep(n)
        B, C = ctx.factors()
        return dict(B=B, C=C, R=ctx.residual(), trace=ctx.trace(), f=ctx.objective(), info=ctx.info())


# one CTA; K = 1; more CTAs than row slices; long columns, one a CTA; a ragged last CTA; near the capacity
SHAPES = [(5, 7, 2), (40, 16, 1), (3, 3000, 1), (200, 1000, 10), (33, 2433, 7), (4099, 150, 5), (9000, 450, 3),
          (1024, 2414, 25), (513, 9001, 4), (2500, 2401, 6)]


@pytest.mark.parametrize("order", ["hals", "dbcd"])
@pytest.mark.parametrize("M,N,K", SHAPES)
def test_matches_oracle(did, M, N, K, order):
    X, _, _ = W.planted(M, N, K, seed=M + N, sigma=0.05)
    B0, C0 = W.init_factors(M, N, K, 5)
    code = did.DID_ORDER_INTERLEAVED if order == "hals" else did.DID_ORDER_DID
    ref = O.factor(X, B0, C0, order=order, max_iter=6, stop="none")
    got = run(did, X, B0, C0, (1, 5), order=code)
    again = run(did, X, B0, C0, (1, 5), order=code)
    eB, eC = rel(got["B"], ref["B"]), rel(got["C"], ref["C"])
    eF = float(np.max(np.abs(got["trace"] - ref["trace"]) / ref["trace"]))
    print("resident %s M=%d N=%d K=%d grid=%d: relB %.3g relC %.3g relf %.3g" % (
        order, M, N, K, got["info"]["grid_ctas"], eB, eC, eF))
    assert eB <= 1e-5 and eC <= 1e-5 and eF <= 1e-5      # float32 dots and updates: a few 1e-7, with margin
    for key in ("B", "C", "R", "trace"):
        assert np.array_equal(got[key], again[key]), key
    Rd = X.astype(np.float64) - got["B"].astype(np.float64) @ got["C"].astype(np.float64)
    assert np.max(np.abs(got["R"] - Rd)) <= 1e-4 * max(1.0, float(np.abs(X).max()))


@pytest.mark.parametrize("M,N,K,sweeps", [(513, 9001, 5, 12), (513, 9001, 7, 12), (300, 9601, 3, 20), (1040, 4961, 3, 20)])
def test_odd_k_sweeps_of_one_launch(did, M, N, K, sweeps):
    """With odd K the last step of a sweep keeps its row of C in the buffer the
    update before it reads: rows that some warps of a CTA have more of than
    others (ld not a multiple of 512), and more than 32 columns a CTA."""
    X, _, _ = W.planted(M, N, K, seed=M + K, sigma=0.05)
    B0, C0 = W.init_factors(M, N, K, 5)
    ref = O.factor(X, B0, C0, order="hals", max_iter=sweeps, stop="none")
    got = run(did, X, B0, C0, (sweeps,))
    assert -(-N // got["info"]["grid_ctas"]) > 32
    assert rel(got["B"], ref["B"]) <= 1e-5 and rel(got["C"], ref["C"]) <= 1e-5
    for _ in range(3):
        again = run(did, X, B0, C0, (sweeps,))
        for key in ("B", "C", "R", "trace"):
            assert np.array_equal(got[key], again[key]), key
    # each step of a sweep rounds an entry of R three times, by 2^-24 of |R| and of the product each
    S = np.abs(got["B"]).astype(np.float64) @ got["C"].astype(np.float64)
    Rd = X.astype(np.float64) - got["B"].astype(np.float64) @ got["C"].astype(np.float64)
    assert np.all(np.abs(got["R"] - Rd) <= 3 * K * sweeps * 2.0 ** -24 * (np.abs(X) + S))


@pytest.mark.parametrize("order", [0, 1])
def test_bfloat16_residual_and_refresh(did, order):
    M, N, K = 700, 1501, 12
    X, _, _ = W.planted(M, N, K, seed=9, sigma=0.05)
    B0, C0 = W.init_factors(M, N, K, 5)
    ref = O.factor(X, B0, C0, order="dbcd" if order else "hals", max_iter=6, stop="none")
    got = run(did, X, B0, C0, (6,), order=order, precision=did.DID_BF16R, refresh_every=4)
    assert got["info"]["refreshes"] == 1
    assert abs(got["f"] - ref["trace"][-1]) <= 1e-3 * ref["trace"][-1]


def test_zero_norm_and_paper_rule(did):
    M, N, K = 60, 500, 4
    X, _, _ = W.planted(M, N, K, seed=1, sigma=0.05)
    B0, C0 = W.init_factors(M, N, K, 2)
    C0[2] = 0.0
    B0[:, 1] = 0.0
    for order, code in (("hals", 0), ("dbcd", 1)):
        ref = O.factor(X, B0, C0, order=order, max_iter=5, stop="none")
        got = run(did, X, B0, C0, (5,), order=code)
        assert got["info"]["degenerate_events"] >= 1
        assert rel(got["B"], ref["B"]) <= 1e-5 and rel(got["C"], ref["C"]) <= 1e-5


def test_static_call_takes_it(did):
    torch = pytest.importorskip("torch")
    M, N, K = 130, 777, 5
    X, _, _ = W.planted(M, N, K, seed=4, sigma=0.05)
    B0, C0 = W.init_factors(M, N, K, 4)
    ref = O.factor(X, B0, C0, order="hals", max_iter=4, stop="none")
    ld = 132
    R = torch.zeros((N, ld), device="cuda")
    R[:, :M] = torch.from_numpy(np.ascontiguousarray((X - (B0.astype(np.float64) @ C0)).T.astype(np.float32))).cuda()
    B = torch.zeros((K, ld), device="cuda")
    B[:, :M] = torch.from_numpy(np.ascontiguousarray(B0.T)).cuda()
    C = torch.from_numpy(C0).cuda()
    for n in (3, 1):                    # the scratch array keeps the first call's words
        did.did_sweep_static(R, ld, B, C, M, N, K, n)
    assert rel(B[:, :M].cpu().numpy().T, ref["B"]) <= 1e-5 and rel(C.cpu().numpy(), ref["C"]) <= 1e-5
    assert float(R[:, M:].abs().max()) == 0.0


@pytest.mark.parametrize("M,N", [(200, 30001), (530, 9001), (16, 100003)])
def test_objective_of_large_and_small_columns(did, M, N):
    """1/2 ||R||^2 where the first column of each CTA's range is far larger than
    the others: squares are added four columns at a time in float32 and then as
    pairs.  (One float32 chain over a CTA's columns was 2.4e-8 to 1.1e-7 off.)"""
    rng = np.random.default_rng(M)
    Xt = rng.random((N, M)).astype(np.float32)
    with did.Context(Xt, M, N, 1, seed=1) as ctx:
        nc = -(-N // ctx.info()["grid_ctas"])
    Xt[::nc] = (1e4 * (0.9 + 0.1 * rng.random(Xt[::nc].shape))).astype(np.float32)
    with did.Context(Xt, M, N, 1, B_init=np.full((1, M), 1e-3, np.float32), C_init=np.full((1, N), 1e-3, np.float32),
                     grid_ctas=0) as ctx:
        assert ctx.info()["sweep_form"] == did.DID_FORM_RESIDENT and -(-N // ctx.info()["grid_ctas"]) == nc
        ctx.sweep(1)
        f, R = ctx.trace()[-1], ctx.residual().astype(np.float64)
    fd = 0.5 * float(np.sum(R * R))
    print("M=%d N=%d nc=%d: %.3g" % (M, N, nc, abs(f - fd) / fd))
    # four roundings of up to 2^-24 of a thread's four squares, of random sign: over some 10^4 groups of
    # large entries that is about 2^-24 / 100
    assert abs(f - fd) <= 1e-8 * fd
