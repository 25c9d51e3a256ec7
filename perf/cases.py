"""What the framework's speed is measured on: calls of its public Python API, as
a user's program makes them, over the sizes, orders and precisions that the
repository's workloads, tests and benchmark use.

A case is one pass of one kind of call:

  solve    a whole factorisation of a matrix on the GPU: create, sweep, read
           the factors and the trace, destroy -- what a script that factors
           one matrix does (the small planted workload).
  sweep    further sweeps of a context that is kept, then the factors and the
           objective -- the inner part of a long factorisation (the
           tall-and-wide, image-like and salt workloads; all block orders).
  static   sweeps on caller-owned R, B and C without any device allocation.
  resume   a checkpoint restored into a kept context: set the factors, form the
           residual anew, read it, evaluate the exact objective.
  serve    a batch of requests of mixed sizes through the serving loop.

Inputs: "uniform" X = B0 C0 + 0.01 |N(0,1)| with B0, C0 ~ U[0,1); "exp" the same
with C0 ~ Exp(1), 30 % zeros, and noise 0.05; "salt" B0 C0 with 1 % of the entries set
to 5.0; "image" 80 % exact zeros, the rest Beta(2,2).
"""

import math
import random

import numpy as np
import torch

import paper_1802_08938_gb300 as did

ORDERS = {"interleaved": did.DID_ORDER_INTERLEAVED, "did": did.DID_ORDER_DID, "batched": did.DID_ORDER_DID_BATCHED}
PRECISIONS = {"fp32": did.DID_FP32, "bf16r": did.DID_BF16R}

# On-chip bytes (L2 and the SMs' shared memory) of a GB300: a residual larger
# than this has to be read from HBM once for each block it is contracted with.
ON_CHIP = 160e6


def case(kind, M, N, K, name=None, data="uniform", precision="fp32", order="interleaved", sweeps=1, refresh=0,
         inner=1, requests=0, mix=0, scale=False):
    c = dict(kind=kind, M=M, N=N, K=K, data=data, precision=precision, order=order, sweeps=sweeps, refresh=refresh,
             inner=inner, requests=requests, mix=mix, scale=scale)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest workload: 100 sweeps of a 200 x 1000 matrix, bound by latency
        case("solve", 200, 1000, 10, "solve_200x1000_k10", sweeps=100),
        # a face-image-sized matrix (1024 pixels, 2414 samples) with the bfloat16 residual
        case("solve", 1024, 2414, 25, "solve_1024x2414_k25_bf16r", precision="bf16r", sweeps=40, refresh=5),
        # sweeps inside a program that owns all device memory
        case("static", 1024, 2414, 25, "static_1024x2414_k25", sweeps=5),
        # image-like data: short columns, many samples; in both precisions
        case("sweep", 784, 70000, 16, "sweep_784x70000_k16", data="image", sweeps=5, scale=True),
        case("sweep", 784, 70000, 16, "sweep_784x70000_k16_bf16r", data="image", precision="bf16r", sweeps=5,
             refresh=10, scale=True),
        # the benchmark's tall-and-wide workload, the largest float32 one
        case("sweep", 5000, 200000, 50, "sweep_5000x200000_k50", data="exp", sweeps=2, refresh=10),
        # the precision workload on a fifth of its samples
        case("sweep", 10000, 100000, 100, "sweep_10000x100000_k100_bf16r", data="salt", precision="bf16r", sweeps=1,
             refresh=5),
        # a term-document-sized matrix in the paper's own block order, per k
        case("sweep", 8165, 18821, 20, "cfirst_8165x18821_k20", data="exp", order="did", sweeps=2),
        # the paper's Algorithm 3 with one reduction per sweep, plain and with inner repeats
        case("sweep", 5000, 200000, 50, "batched_5000x200000_k50", data="exp", order="batched", sweeps=4),
        case("sweep", 784, 70000, 16, "batched_784x70000_k16_inner2", data="image", order="batched", sweeps=5, inner=2,
             scale=True),
        # restore, residual and exact objective, with a number of factors beyond 64
        case("resume", 8165, 18821, 100, "resume_8165x18821_k100", data="exp"),
        # serving: requests of 64..4096 rows and 256..65536 samples at once
        case("serve", 4096, 65536, 64, "serve_24", requests=24, mix=1, sweeps=20),
    ]


def logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "static", "sweep", "sweep", "sweep", "resume", "serve"])
    precision = rng.choice(["fp32", "bf16r"])
    if kind == "solve":
        M, N = logint(rng, 32, 2048), logint(rng, 64, 8192)
        K = rng.randint(2, min(32, M, N))
        order = rng.choice(["interleaved", "interleaved", "did", "batched"])
        return case(kind, M, N, K, precision="fp32" if order == "batched" else precision, order=order,
                    sweeps=rng.randint(10, 60), refresh=rng.choice([0, 5, 10]))
    if kind == "static":
        M, N = logint(rng, 64, 4096), logint(rng, 256, 32768)
        return case(kind, M, N, rng.randint(4, 32), sweeps=rng.randint(1, 5))
    if kind == "sweep":
        M = logint(rng, 200, 10000)
        N = logint(rng, 2000, min(200000, 10 ** 9 // M))
        order = rng.choice(["interleaved", "interleaved", "interleaved", "did", "batched"])
        K = rng.randint(4, 64 if order == "batched" else 100)
        data = rng.choice(["uniform", "exp", "salt", "image"])
        return case(kind, M, N, K, data=data, precision="fp32" if order == "batched" else precision, order=order,
                    sweeps=1, refresh=rng.choice([0, 5, 10]), inner=rng.choice([1, 2]) if order == "batched" else 1,
                    scale=data == "image")
    if kind == "resume":
        M = logint(rng, 200, 10000)
        N = logint(rng, 2000, min(60000, 2 * 10 ** 8 // M))
        return case(kind, M, N, rng.randint(4, 128), data=rng.choice(["uniform", "exp"]), precision=precision)
    return case(kind, 4096, 65536, 64, precision=precision, requests=rng.randint(4, 24), mix=rng.randrange(1 << 20),
                sweeps=rng.randint(5, 20))


# ------------------------------------------------------------------- inputs
def planted(M, N, K, data, seed):
    """X as an (N, M) float32 tensor on the GPU (M x N column-major)."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    X = torch.empty((N, M), dtype=torch.float32, device="cuda")
    step = max(1, (1 << 28) // M)
    if data == "image":
        for j in range(0, N, step):
            n = min(step, N - j)
            u = torch.rand((3, n, M), generator=g, device="cuda").median(dim=0).values       # Beta(2,2)
            keep = torch.rand((n, M), generator=g, device="cuda") >= 0.8
            X[j:j + n] = u * keep
        return X
    B0 = torch.rand((K, M), generator=g, device="cuda")
    C0 = torch.rand((K, N), generator=g, device="cuda")
    if data == "exp":
        C0 = -torch.log1p(-C0) * (torch.rand((K, N), generator=g, device="cuda") >= 0.3)
    sigma = {"uniform": 0.01, "exp": 0.05, "salt": 0.0}[data]
    torch.mm(C0.t(), B0, out=X)
    for j in range(0, N, step):
        n = min(step, N - j)
        if sigma:
            X[j:j + n] += sigma * torch.randn((n, M), generator=g, device="cuda").abs()
        if data == "salt":
            X[j:j + n][torch.rand((n, M), generator=g, device="cuda") < 0.01] = 5.0
    return X


def mix_shapes(c):
    """(M, N, K) of each request of the mix: M, N log-uniform, K from {8, 16, 32, 64}."""
    r = random.Random(c["mix"])
    return [(logint(r, 64, c["M"]), logint(r, 256, c["N"]), r.choice((8, 16, 32, 64))) for _ in range(c["requests"])]


def factors_like(M, N, K, seed):
    """Factors a checkpoint might hold: (K, M) and (K, N), float32, on the GPU."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.rand((K, M), generator=g, device="cuda"), torch.rand((K, N), generator=g, device="cuda")


def options(c):
    return dict(precision=PRECISIONS[c["precision"]], order=ORDERS[c["order"]], refresh_every=c["refresh"],
                init_scale=c["scale"], inner_c=c["inner"], inner_b=c["inner"])


def start_seed(seed):
    return seed % 1000003


# ------------------------------------------------------------------ the calls
def prepare(c, seed):
    M, N, K = c["M"], c["N"], c["K"]
    s = dict(c=c, seed=start_seed(seed))
    if c["kind"] == "serve":
        s["X"] = [planted(m, n, k, "uniform", 1000 * seed + i) for i, (m, n, k) in enumerate(mix_shapes(c))]
        s["server"] = did.Server(32 << 30, precision=PRECISIONS[c["precision"]], max_slots=64)
        return s
    X = planted(M, N, K, c["data"], seed)
    if c["kind"] == "solve":
        s["X"] = X
        return s
    if c["kind"] == "static":
        ld = (M + 3) // 4 * 4
        B, C = factors_like(M, N, K, seed + 1)
        s["ld"] = ld
        s["B"] = torch.zeros((K, ld), device="cuda")
        s["B"][:, :M] = B
        s["C"] = C
        s["R"] = torch.zeros((N, ld), device="cuda")
        s["R"][:, :M] = X - C.t() @ B
        s["trace"] = torch.empty(c["sweeps"], dtype=torch.float64, device="cuda")
        return s
    s["ctx"] = did.Context(X, M, N, K, seed=s["seed"], **options(c))
    s["B"] = torch.empty((K, M), device="cuda")
    s["C"] = torch.empty((K, N), device="cuda")
    if c["kind"] == "resume":
        s["B0"], s["C0"] = factors_like(M, N, K, seed + 1)
        s["R"] = torch.empty((N, M), device="cuda")
    return s


def run(s):
    c = s["c"]
    M, N, K = c["M"], c["N"], c["K"]
    if c["kind"] == "solve":
        with did.Context(s["X"], M, N, K, seed=s["seed"], **options(c)) as ctx:
            ctx.factor(c["sweeps"], 0.0)
            B, C = ctx.factors()
            return {"B": B, "C": C, "trace": ctx.trace()}
    if c["kind"] == "static":
        did.did_sweep_static(s["R"], s["ld"], s["B"], s["C"], M, N, K, c["sweeps"], trace=s["trace"])
        return {"R": s["R"], "B": s["B"], "C": s["C"], "trace": s["trace"]}
    if c["kind"] == "serve":
        srv = s["server"]
        tickets = [srv.submit(m, n, k, s["seed"] + i, max_iter=c["sweeps"], tol=0.0, X=s["X"][i])
                   for i, (m, n, k) in enumerate(mix_shapes(c))]
        objs, out = [], []
        for t in tickets:
            objs.append(srv.wait(t)["obj"])
            out.append(srv.fetch(t))
        return {"factors": out, "objective": np.array(objs)}
    ctx = s["ctx"]
    if c["kind"] == "resume":
        did.did_set_factors(ctx.h, s["B0"], s["C0"])
        did.did_get_residual(ctx.h, s["R"])
        return {"R": s["R"], "residual_objective": ctx.residual_objective(), "objective": ctx.objective()}
    ctx.sweep(c["sweeps"])
    did.did_get_factors(ctx.h, s["B"], s["C"])
    # the trace of a bfloat16 residual reads a few percent high, so there a
    # program asks for the exact f(B, C)
    f = ctx.objective() if c["precision"] == "bf16r" else ctx.residual_objective()
    return {"B": s["B"], "C": s["C"], "objective": f}


# --------------------------------------------------------------- what it needs
def work(c):
    """Bytes and operations a pass cannot do without.  A sweep of the rank-one
    orders contracts the residual with each c_k and each b_k, 4 M N K
    operations, and applies the changes, another 4 M N K.  A residual that fits on the
    chip is read and written once; a larger one is read once per k (c_k needs
    every earlier block; twice per k in the C-first order, whose B step follows its C step) and written once
    per sweep.  The batched order reads R for g and reads and writes it for
    the update."""
    elem = 2 if c["precision"] == "bf16r" else 4
    if c["kind"] == "serve":
        b = f = 0.0
        for m, n, k in mix_shapes(c):
            r = m * n * elem
            b += m * n * 4 + (c["sweeps"] * (k + 1) * r if r > ON_CHIP else 2 * r) + 4.0 * k * (m + n)
            f += 8.0 * m * n * k * c["sweeps"]
        return {"bytes": b, "flops": f}
    M, N, K = c["M"], c["N"], c["K"]
    R, F = float(M) * N * elem, 4.0 * K * (M + N)
    if c["kind"] == "resume":
        # X read and R written; R read and copied out; X read for the objective
        return {"bytes": 8.0 * M * N + 2 * R + 4.0 * M * N + 2 * F, "flops": 4.0 * M * N * K}
    n = c["sweeps"]
    if c["order"] == "batched":
        b = n * 3 * R
    elif R <= ON_CHIP:
        b = 2 * R
    else:
        b = n * (K * (2 if c["order"] == "did" else 1) + 1) * R
    if c["kind"] == "solve" or (c["kind"] == "sweep" and c["precision"] == "bf16r"):
        b += 4.0 * M * N
    return {"bytes": b + 2 * F, "flops": 8.0 * M * N * K * n}


def tolerance(c):
    """Measured against the 64-bit values and against runs with another grid
    (sums in another order), on the listed and some twenty drawn cases; about four times the largest seen.
    float32: factors up to 2.5e-6 from 64 bits, the residual of a restored
    checkpoint 6e-7.  bfloat16 residual: its storage moves factors by up to
    1e-2 (short image-like columns; 2e-4 to 1e-3 mostly), a rounded residual
    by 1.7e-3, f(B, C) by less."""
    if c["precision"] == "bf16r":
        return {"rel": 7e-3, "max": 0.05} if c["kind"] == "resume" else {"rel": 3e-2, "max": 0.5}
    return {"rel": 2.5e-6} if c["kind"] == "resume" else {"rel": 1e-5}


# ------------------------------------------------- the same in 64 bits, in torch
def splitmix_uniform(n, seed, stream):
    """n float32 uniforms of the library's counter-based generator (SplitMix64)."""
    def mix(z):
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return z ^ (z >> np.uint64(31))
    golden = np.uint64(0x9E3779B97F4A7C15)
    with np.errstate(over="ignore"):
        key = mix(np.array([seed], np.uint64) + np.uint64(stream + 1) * golden)
        w = mix(key + (np.arange(n, dtype=np.uint64) + np.uint64(1)) * golden)
    return (w >> np.uint64(40)).astype(np.float64) * 2.0 ** -24


def start64(X, M, N, K, seed, scale):
    B = torch.from_numpy(splitmix_uniform(M * K, seed, 4).reshape(K, M)).cuda()
    C = torch.from_numpy(splitmix_uniform(K * N, seed, 5).reshape(K, N)).cuda()
    if scale:
        a = ((X @ B.t()) * C.t()).sum() / ((B @ B.t()) * (C @ C.t())).sum()
        f = a.sqrt().float()
        B, C = (B.float() * f).double(), (C.float() * f).double()
    return B, C


def step_b(R, B, C, k):
    c = C[k]
    cc = c @ c
    if cc > 0:
        b = (B[k] + (c @ R) / cc).clamp_(min=0)
        R.addr_(c, B[k] - b)
        B[k] = b


def step_c(R, B, C, k):
    b = B[k]
    bb = b @ b
    if bb > 0:
        c = (C[k] + (R @ b) / bb).clamp_(min=0)
        R.addr_(C[k] - c, b)
        C[k] = c


def sweeps64(R, B, C, order, n, inner=1):
    """n sweeps on R = (X - B C)^T in place; the objectives after each."""
    K, f = B.shape[0], []
    for _ in range(n):
        if order == "interleaved":
            for k in range(K):
                step_b(R, B, C, k)
                step_c(R, B, C, k)
        else:
            for step in (step_c, step_b):
                for _ in range(inner):
                    for k in range(K):
                        step(R, B, C, k)
        f.append(0.5 * float((R * R).sum()))
    return f


def exact(c, seed):
    M, N, K = c["M"], c["N"], c["K"]
    s0 = start_seed(seed)
    if c["kind"] == "serve":
        objs, out = [], []
        for i, (m, n, k) in enumerate(mix_shapes(c)):
            X = planted(m, n, k, "uniform", 1000 * seed + i).double()
            B, C = start64(X, m, n, k, s0 + i, False)
            objs.append(sweeps64(X.addmm_(C.t(), B, alpha=-1), B, C, "interleaved", c["sweeps"])[-1])
            out.append((B.t().contiguous().cpu().numpy(), C.cpu().numpy()))
        return {"factors": out, "objective": np.array(objs)}
    X = planted(M, N, K, c["data"], seed).double()
    if c["kind"] == "resume":
        B, C = (t.double() for t in factors_like(M, N, K, seed + 1))
        R = X.addmm_(C.t(), B, alpha=-1)
        f = 0.5 * float((R * R).sum())
        return {"R": R, "residual_objective": f, "objective": f}
    if c["kind"] == "static":
        Bf, Cf = factors_like(M, N, K, seed + 1)
        ld = (M + 3) // 4 * 4
        R = torch.zeros((N, ld), dtype=torch.float64, device="cuda")
        R[:, :M] = (X.float() - Cf.t() @ Bf).double()
        B = torch.zeros((K, ld), dtype=torch.float64, device="cuda")
        B[:, :M] = Bf.double()
        C = Cf.double()
        f = sweeps64(R, B, C, "interleaved", c["sweeps"])
        return {"R": R, "B": B, "C": C, "trace": torch.tensor(f, dtype=torch.float64)}
    B, C = start64(X, M, N, K, s0, c["scale"])
    R = X.addmm_(C.t(), B, alpha=-1)
    f0 = 0.5 * float((R * R).sum())
    f = sweeps64(R, B, C, c["order"], c["sweeps"], c["inner"])
    if c["kind"] == "solve":
        return {"B": B.t().contiguous().cpu().numpy(), "C": C.cpu().numpy(), "trace": np.array([f0] + f)}
    return {"B": B, "C": C, "objective": f[-1]}
