"""Read-only sweeps of the interleaved order: R keeps its value for a sweep,
the changes stay pending, and R is formed anew on the tensor cores after it.

Shapes beyond the SMs' shared memory, one for each way a column is held
(threads of a group 32 to 512, one to ten vectors a thread), with column
counts that leave part of a chunk, of a round of the groups and of a unit.
Against the FP64 oracle's HALS sweeps and the kernel that writes R for every k.
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
        ctx.sweep(sweeps)
        B, C = ctx.factors()
        return dict(B=B, C=C, R=ctx.residual(), trace=ctx.trace(), f=ctx.objective(), info=ctx.info())


SHAPES = [(64, 150001, 16), (130, 70003, 7), (784, 12001, 5), (1030, 9001, 2), (2064, 4503, 9), (5003, 1999, 3),
          (9000, 1051, 1), (12000, 801, 4), (14001, 641, 2), (16001, 601, 3), (17001, 541, 2),
          (600, 16001, 65), (1100, 9005, 101), (520, 20011, 128)]


@pytest.mark.parametrize("M,N,K", SHAPES)
def test_float32_matches_oracle(did, M, N, K):
    X, _, _ = W.planted(M, N, K, seed=M + N, sigma=0.05)
    B0, C0 = W.init_factors(M, N, K, 5)
    ref = O.factor(X, B0, C0, order="hals", max_iter=3, stop="none")
    got = run(did, X, B0, C0, 3)
    assert got["info"]["sweep_form"] == did.DID_FORM_READ_ONLY and got["info"]["pass_blocks"] == 1
    again = run(did, X, B0, C0, 3)
    eager = run(did, X, B0, C0, 3, flags=did.DID_FLAG_EAGER_WRITEBACK)
    eB, eC = rel(got["B"], ref["B"]), rel(got["C"], ref["C"])
    eF = float(np.max(np.abs(got["trace"] - ref["trace"]) / ref["trace"]))
    print("read-only M=%d N=%d K=%d GS=%d NR=%d: relB %.3g relC %.3g relf %.3g (eager %.3g %.3g)" % (
        M, N, K, got["info"]["group_threads"], got["info"]["vecs_per_thread"], eB, eC, eF, rel(eager["B"], ref["B"]),
        rel(eager["C"], ref["C"])))
    # float32 dots over up to 150001 terms and the refresh's 2^-21 |B||C|: a few 1e-7 each, 1e-5 with margin
    assert eB <= 1e-5 and eC <= 1e-5 and eF <= 1e-5
    assert np.array_equal(got["B"], again["B"]) and np.array_equal(got["C"], again["C"])
    assert np.array_equal(got["trace"], again["trace"])
    Rd = X.astype(np.float64) - got["B"].astype(np.float64) @ got["C"].astype(np.float64)
    S = np.abs(got["B"]).astype(np.float64) @ got["C"].astype(np.float64)
    assert np.all(np.abs(got["R"] - Rd) <= 2.0 ** -17 * S + 2.0 ** -22 * np.abs(Rd) + 1e-6)


@pytest.mark.parametrize("M,N,K", [(18001, 541, 2), (600, 16001, 129), (120, 70003, 33)])
def test_shapes_that_keep_the_kernel_that_writes_r(did, M, N, K):
    """Columns of which the ring holds no three, more than 128 blocks, and
    blocks too many for their column: the general kernel, without a flag."""
    X, _, _ = W.planted(M, N, K, seed=M + N, sigma=0.05)
    B0, C0 = W.init_factors(M, N, K, 5)
    ref = O.factor(X, B0, C0, order="hals", max_iter=2, stop="none")
    got = run(did, X, B0, C0, 2)
    assert got["info"]["sweep_form"] == did.DID_FORM_WRITING and got["info"]["pass_blocks"] == 0
    assert rel(got["B"], ref["B"]) <= 1e-5 and rel(got["C"], ref["C"]) <= 1e-5


@pytest.mark.parametrize("M,N,K", [(130, 70003, 7), (784, 12001, 20), (2064, 4503, 9), (9000, 1051, 70), (16001, 601, 4),
                                   (17001, 541, 3), (520, 20011, 128)])
def test_bfloat16_residual(did, M, N, K):
    X, _, _ = W.planted(M, N, K, seed=M + N, sigma=0.05)
    B0, C0 = W.init_factors(M, N, K, 5)
    ref = O.factor(X, B0, C0, order="hals", max_iter=3, stop="none")
    got = run(did, X, B0, C0, 3, precision=did.DID_BF16R, refresh_every=2)
    assert got["info"]["sweep_form"] == did.DID_FORM_READ_ONLY
    assert got["info"]["refreshes"] == 1
    eB, eC = rel(got["B"], ref["B"]), rel(got["C"], ref["C"])
    print("read-only bfloat16 M=%d N=%d K=%d: relB %.3g relC %.3g" % (M, N, K, eB, eC))
    # R is rounded by up to 2^-9 of an entry once a sweep; a contraction carries at most that share of |R| |c|
    assert eB <= 3 * 2.0 ** -9 and eC <= 3 * 2.0 ** -9
    assert abs(got["f"] - ref["trace"][-1]) <= 1e-3 * ref["trace"][-1]


def test_stopping_zero_norms_and_resume(did):
    M, N, K = 800, 12003, 4
    X, _, _ = W.planted(M, N, K, seed=1, sigma=0.05)
    B0, C0 = W.init_factors(M, N, K, 2)
    C0[2] = 0.0                         # ||c_3|| = 0: b_3 is left unchanged until c_3 is updated
    ref = O.factor(X, B0, C0, order="hals", max_iter=60, tol=1e-2, stop="relchange")
    Xc = np.ascontiguousarray(X.T)
    with did.Context(Xc, M, N, K, B_init=np.ascontiguousarray(B0.T), C_init=C0) as ctx:
        assert ctx.info()["sweep_form"] == did.DID_FORM_READ_ONLY
        iters, f = ctx.factor(60, 1e-2)
        B, C = ctx.factors()
        assert iters == ref["iters"] and ctx.info()["degenerate_events"] >= 1
        assert rel(B, ref["B"]) <= 1e-5 and rel(C, ref["C"]) <= 1e-5
        ctx.sweep(2)
        B1, C1 = ctx.factors()
        ctx.set_factors(B, C)
        ctx.sweep(2)
        B2, C2 = ctx.factors()
    assert rel(B2, B1) <= 1e-5 and rel(C2, C1) <= 1e-5


def test_expired_wait_is_reported(did):
    M, N, K = 800, 12003, 3
    X, _, _ = W.planted(M, N, K, seed=1, sigma=0.05)
    with did.Context(np.ascontiguousarray(X.T), M, N, K, seed=0, timeout_ns=10 ** 7, debug_barrier_extra=1) as ctx:
        with pytest.raises(did.DIDError) as e:
            ctx.sweep(1)
        assert e.value.status == did.DID_ETIMEOUT
        B, C = ctx.factors()
        assert np.isfinite(B).all() and (B >= 0).all() and np.isfinite(C).all() and (C >= 0).all()


@pytest.mark.parametrize("M,N,K,grid", [(2048, 2105, 4, 1), (4096, 1101, 3, 2), (2064, 2100, 4, 1), (3000, 2000, 4, 1),
                                        (5000, 1000, 4, 2), (9000, 600, 3, 4)])
def test_few_ctas(did, M, N, K, grid):
    """A grid given by the caller: slices of 2048 rows, the longest that phase A
    of the read-only sweep adds up, and longer ones, which the kernel that
    writes R takes."""
    X, _, _ = W.planted(M, N, K, seed=M + N, sigma=0.05)
    B0, C0 = W.init_factors(M, N, K, 5)
    ref = O.factor(X, B0, C0, order="hals", max_iter=3, stop="none")
    got = run(did, X, B0, C0, 3, grid_ctas=grid)
    assert got["info"]["grid_ctas"] == grid
    rows = -(-((M + 15) // 16 * 16) // grid)
    assert got["info"]["sweep_form"] == (did.DID_FORM_READ_ONLY if rows <= 2048 else did.DID_FORM_WRITING)
    eB, eC = rel(got["B"], ref["B"]), rel(got["C"], ref["C"])
    eF = float(np.max(np.abs(got["trace"] - ref["trace"]) / ref["trace"]))
    print("read-only M=%d N=%d K=%d grid=%d: relB %.3g relC %.3g relf %.3g" % (M, N, K, grid, eB, eC, eF))
    assert eB <= 1e-5 and eC <= 1e-5 and eF <= 1e-5


def test_expired_wait_ends_the_queued_sweeps(did):
    """After an expired wait the sweeps queued behind it change nothing: B and C
    are those that one sweep leaves, whatever the number asked for, and the
    context goes on from them."""
    M, N, K = 800, 12003, 3
    X, _, _ = W.planted(M, N, K, seed=1, sigma=0.05)
    left = []
    for n in (1, 6, 6):
        with did.Context(np.ascontiguousarray(X.T), M, N, K, seed=0, timeout_ns=10 ** 7, debug_barrier_extra=1) as ctx:
            with pytest.raises(did.DIDError) as e:
                ctx.sweep(n)
            assert e.value.status == did.DID_ETIMEOUT
            left.append((*ctx.factors(), ctx.trace(), ctx.info()["sweeps_done"]))
    for B, C, trace, done in left[1:]:
        assert np.array_equal(B, left[0][0]) and np.array_equal(C, left[0][1])
        assert len(trace) == 1 and done == 0


@pytest.mark.parametrize("order,K", [(0, 1), (1, 1), (0, 70)])
def test_stop_ends_the_queued_sweeps(did, order, K):
    """With a stopping rule a few sweeps are queued ahead.  Once it holds, the
    passes that would form R again do nothing either: a call that stops after
    its first sweep takes no longer than one sweep (three more passes over X and R
    would triple it at K = 1), and the next call goes on from the same state."""
    M, N = (1500, 40000) if K == 1 else (300, 40000)
    X, _, _ = W.planted(M, N, K, seed=3, sigma=0.05)
    Xc = np.ascontiguousarray(X.T)
    with did.Context(Xc, M, N, K, seed=1, order=order) as a, did.Context(Xc, M, N, K, seed=1, order=order) as b:
        ms = {}
        for ctx, call in ((a, lambda: a.sweep(1)), (b, lambda: b.factor(4, 1.0))):
            t = []
            for _ in range(6):
                t0 = ctx.info()["sweep_kernel_ms"]
                call()
                t.append(ctx.info()["sweep_kernel_ms"] - t0)
            ms[ctx] = min(t)
        assert a.info()["sweeps_done"] == 6 and b.info()["sweeps_done"] == 6
        for x, y in zip((*a.factors(), a.trace(), a.residual()), (*b.factors(), b.trace(), b.residual())):
            assert np.array_equal(x, y)
        print("order %d K=%d: one sweep %.3f ms, stopped after one %.3f ms" % (order, K, ms[a], ms[b]))
        if K == 1:
            assert ms[b] <= 2.0 * ms[a]      # queued launches that return at once; 2.6 and 3.0 with the passes


@pytest.mark.parametrize("order", [0, 1])
@pytest.mark.parametrize("precision,share", [(0, 2.0 ** -42), (1, 2.0 ** -32)])
def test_exact_fit_settles_at_the_refresh_error(did, order, precision, share):
    """A noise-free rank-one matrix.  R is formed anew in each sweep, so f settles
    where the refresh's error leaves it: 2^-21 of |B||C| an entry (2^-16 for a
    bfloat16 residual), squared and halved."""
    M, N = 800, 12003
    X, _, _ = W.planted(M, N, 1, seed=3, sigma=0.0)
    xx = float(np.sum(X.astype(np.float64) ** 2))
    with did.Context(np.ascontiguousarray(X.T), M, N, 1, seed=1, order=order, precision=precision) as ctx:
        assert ctx.info()["sweep_form"] == did.DID_FORM_READ_ONLY
        ctx.sweep(60)
        f, trace = ctx.objective(), ctx.trace()
    print("exact fit order %d precision %d: f %.3g, trace %.3g of ||X||^2" % (order, precision, f / xx, trace[-1] / xx))
    assert f <= 0.5 * share * xx and trace[-1] <= 0.5 * share * xx


def test_no_room_for_the_scratch(did):
    """Where the pending factors (102 MB) do not fit on the device beside X, R and
    C, the context takes the kernel that writes R."""
    torch = pytest.importorskip("torch")
    M, N, K = 520, 200003, 128
    X = torch.empty((N, M), device="cuda")
    did.did_generate_planted(X, M, N, K, 5, sigma=0.05)

    def factors(**kw):
        with did.Context(X, M, N, K, seed=2, **kw) as ctx:
            ctx.sweep(1)
            i = ctx.info()
            return (*ctx.factors(), i["sweep_form"], i["device_bytes"])

    with_room = factors()
    writing = factors(flags=did.DID_FLAG_LAZY_WRITEBACK)     # what a float32 residual runs without a flag then
    assert with_room[2] == did.DID_FORM_READ_ONLY and with_room[3] - writing[3] >= 100 << 20
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    ballast = torch.empty(free - writing[3] - (60 << 20), dtype=torch.uint8, device="cuda")
    try:
        got = factors()
    finally:
        del ballast
        torch.cuda.empty_cache()
    assert got[2] == did.DID_FORM_WRITING and got[3] < with_room[3]
    assert np.array_equal(got[0], writing[0]) and np.array_equal(got[1], writing[1])
