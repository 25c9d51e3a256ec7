"""The forms in which the serving loop sweeps its requests: resident in shared
memory, read-only on the whole GPU, and in the multi-instance kernel, with a
mid-sized request going from the last to the second once it is alone.

Each request of the mix against the FP64 oracle and against itself alone.
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


# M, N, K, sweeps: resident (ragged, one CTA and many), mid-sized (just above what is
# resident; the second outlives the others), read-only, and a K too large for its column
MIX = [(33, 257, 3, 4), (300, 9001, 8, 4), (701, 12007, 8, 3), (703, 12001, 7, 12), (699, 12003, 5, 4),
       (1100, 30007, 4, 3), (100, 90001, 30, 2)]


@pytest.mark.parametrize("precision", ["fp32", "bf16r"])
def test_mix_of_forms(did, precision):
    prec = did.DID_FP32 if precision == "fp32" else did.DID_BF16R
    Xs = [np.ascontiguousarray(W.planted(M, N, K, seed=M + N, sigma=0.05)[0].T.astype(np.float32)) for M, N, K, _ in MIX]

    def serve(which):
        out = {}
        with did.Server(8 << 30, precision=prec, max_slots=16, round_sweeps=2) as srv:
            ts = {i: srv.submit(MIX[i][0], MIX[i][1], MIX[i][2], 40 + i, max_iter=MIX[i][3], tol=0.0, X=Xs[i])
                  for i in which}
            for i, t in ts.items():
                r = srv.wait(t)
                assert r["status"] == did.DID_OK and r["iters"] == MIX[i][3]
                out[i] = (*srv.fetch(t), r["obj"])
        return out

    mix = serve(range(len(MIX)))
    alone = serve([3])
    for i, (M, N, K, sweeps) in enumerate(MIX):
        B0, C0 = W.init_factors(M, N, K, 40 + i)
        ref = O.factor(Xs[i].T, B0, C0, order="hals", max_iter=sweeps, stop="none")
        got = [mix[i]] + ([alone[i]] if i in alone else [])
        for B, C, f in got:
            eB, eC, eF = rel(B, ref["B"]), rel(C, ref["C"]), abs(f - ref["trace"][-1]) / ref["trace"][-1]
            print("%s M=%d N=%d K=%d: relB %.3g relC %.3g relf %.3g" % (precision, M, N, K, eB, eC, eF))
            if precision == "fp32":
                # float32 dots and residual, as in the per-context tests
                assert eB <= 1e-5 and eC <= 1e-5 and eF <= 1e-5
            else:
                # a residual rounded to 2^-9 of each entry: the objective of the kept residual to 2^-9 twice over
                assert eF <= 4e-3


def smallest_budget(did, M, N, K):
    """The bytes a server counts for a request: the least budget that takes it."""
    lo, hi = 8 * M * N, 16 * M * N + (64 << 20)
    while hi - lo > 1:
        mid = (lo + hi) // 2
        with did.Server(mid, max_slots=1) as srv:
            try:
                srv.submit(M, N, K, 1, max_iter=1, tol=0.0)
                hi = mid
            except did.DIDError as e:
                assert e.status == did.DID_E_TOO_LARGE
                lo = mid
    return hi


def request(did, M, N, K, seed, sweeps):
    """X of a request on the GPU and the factors that the kernel which writes R gives for it."""
    import torch
    X = torch.empty((N, M), device="cuda")
    did.did_generate_planted(X, M, N, K, 5, sigma=0.05)
    with did.Context(X, M, N, K, seed=seed, flags=did.DID_FLAG_EAGER_WRITEBACK) as ctx:
        ctx.sweep(sweeps)
        return X, ctx.factors()


# resident; read-only (a quarter of X for the pending c, half of it for the refresh's operands)
@pytest.mark.parametrize("M,N,K", [(300, 9001, 8), (256, 200003, 64)])
def test_scratch_stays_in_the_budget(did, M, N, K):
    """A budget of just the request leaves no room for its form's scratch: it
    runs in the multi-instance kernel, and the device holds no more than the budget."""
    import torch
    budget = smallest_budget(did, M, N, K)
    X, (B0, C0) = request(did, M, N, K, 7, 3)
    held = {}
    for b in (8 << 30, budget):
        with did.Server(b, max_slots=2) as srv:
            t = srv.submit(M, N, K, 7, max_iter=3, tol=0.0, X=X)            # also loads the kernels it uses
            assert srv.wait(t)["status"] == did.DID_OK
            B, C = srv.fetch(t)
            assert rel(B, B0) <= 1e-5 and rel(C, C0) <= 1e-5
        with did.Server(b, max_slots=2) as srv:
            torch.cuda.synchronize()
            free, least = torch.cuda.mem_get_info()[0], []
            t = srv.submit(M, N, K, 7, max_iter=500, tol=0.0, X=X)
            while srv.wait(t, timeout_ms=2)["status"] == did.DID_PENDING:
                least.append(torch.cuda.mem_get_info()[0])
            st = srv.stats()
            held[b] = free - min(least)
    print("request %d bytes: device held %d with room, %d without, peak %d" % (budget, held[8 << 30], held[budget],
                                                                               st["peak_bytes"]))
    assert st["peak_bytes"] == budget
    assert held[budget] <= budget + (64 << 20)       # the allocator's pool grows in steps of up to 32 MB


def test_scratch_gives_way_to_a_request(did):
    """Two requests within the budget while the first one's scratch takes the
    second's place: the second is admitted, and both come out right."""
    shapes = [(256, 200003, 64, 40), (256, 60001, 8, 4)]
    budget = sum(smallest_budget(did, M, N, K) for M, N, K, _ in shapes)
    rq = [request(did, M, N, K, 40, n) for M, N, K, n in shapes]
    with did.Server(budget, max_slots=2, round_sweeps=1) as srv:
        ts = []
        for (M, N, K, n), (X, _) in zip(shapes, rq):
            ts.append(srv.submit(M, N, K, 40, max_iter=n, tol=0.0, X=X))
            srv.wait(ts[0], timeout_ms=5)            # the first one's first round begins
        for t, (_, (B0, C0)) in zip(ts, rq):
            assert srv.wait(t)["status"] == did.DID_OK
            B, C = srv.fetch(t)
            eB, eC = rel(B, B0), rel(C, C0)
            print("relB %.3g relC %.3g" % (eB, eC))
            # two float32 forms against each other, over up to 40 sweeps
            assert eB <= 1e-4 and eC <= 1e-4
        assert srv.stats()["peak_bytes"] <= budget
