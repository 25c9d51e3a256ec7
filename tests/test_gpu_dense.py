"""The float32 passes over X - B C: the 128 x 128 tiles of larger matrices at
edges of tiles, chunks of K and vectors, against float64, in both precisions.
"""

import numpy as np
import pytest

from synth import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def did():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1802_08938_gb300 as did
    return did


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("M,N,K", [(100, 19457, 1), (128, 19460, 16), (241, 12001, 17), (500, 5003, 65), (1000, 2563, 100)])
def test_refresh_and_objective(did, M, N, K, precision):
    X, _, _ = W.planted(M, N, K, seed=M + N, sigma=0.05)
    B0, C0 = W.init_factors(M, N, K, 5)
    with did.Context(np.ascontiguousarray(X.T), M, N, K, B_init=np.ascontiguousarray(B0.T), C_init=C0,
                     precision=precision, flags=did.DID_FLAG_SIMT_REFRESH) as ctx:
        R, f0, f = ctx.residual(), ctx.trace()[0], ctx.objective()
    P = B0.astype(np.float64) @ C0.astype(np.float64)
    Rd = X.astype(np.float64) - P
    # a chain of K float32 FMAs and one subtraction; bfloat16: half an ulp of 8 bits
    bound = (K + 2) * 2.0 ** -24 * P + 2.0 ** -24 * np.abs(Rd) + (2.0 ** -8 * np.abs(Rd) if precision else 0.0)
    assert np.all(np.abs(R - Rd) <= bound + 1e-30)
    fd = 0.5 * float(np.sum(Rd ** 2))
    assert abs(f - fd) <= 1e-5 * fd and abs(f0 - fd) <= 1e-5 * fd


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("M,N", [(1, 1), (31, 4501), (33, 9003), (100, 7001), (128, 513), (129, 40), (257, 33), (1024, 300), (1025, 299), (8165, 70)])
def test_residual_copies(did, M, N, precision):
    """The residual to device memory (any 4-byte aligned address) and to the host: the same values."""
    import torch
    X, _, _ = W.planted(M, N, 1, seed=M + N, sigma=0.05)
    with did.Context(np.ascontiguousarray(X.T), M, N, 1, seed=3, precision=precision) as ctx:
        host = ctx.residual()
        buf = torch.full((M * N + 2,), 7.0, device="cuda")
        did.did_get_residual(ctx.h, buf[1:M * N + 1])
    got = buf.cpu().numpy()
    assert got[0] == 7.0 and got[-1] == 7.0
    assert np.array_equal(got[1:-1].reshape(N, M), np.asarray(host).T)


@pytest.mark.parametrize("M,N", [(1024, 4001), (700, 6007)])
def test_objective_sums_four_squares_in_float32(did, M, N):
    """Rows 10^4 times the others where a thread of the 128 x 128 tile has its
    first: only the three squares added to a large one in float32 may be lost
    in it (1.2e-8 of f), not all seven of the thread's rows (2.9e-8)."""
    rng = np.random.default_rng(M)
    Xt = rng.random((N, M)).astype(np.float32)
    rows = np.arange(M)
    large = (rows % 128 < 64) & (rows % 4 == 0)
    Xt[:, large] = (1e4 * (0.8 + 0.2 * rng.random((N, int(large.sum()))))).astype(np.float32)
    with did.Context(Xt, M, N, 1, B_init=np.zeros((1, M), np.float32), C_init=np.zeros((1, N), np.float32),
                     flags=did.DID_FLAG_SIMT_REFRESH) as ctx:
        f0, f = ctx.trace()[0], ctx.objective()
    fd = 0.5 * float(np.sum(Xt.astype(np.float64) ** 2))
    print("M=%d N=%d: %.3g %.3g" % (M, N, abs(f - fd) / fd, abs(f0 - fd) / fd))
    assert abs(f - fd) <= 2e-8 * fd and abs(f0 - fd) <= 2e-8 * fd
