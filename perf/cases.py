"""Workloads of the pre-packed tall-and-skinny GEMM, as its users run them.

A case is a dict of plain values.  ``path`` says which entry point it goes through:

* ``execute``  one problem, B packed once and a plan kept: C = alpha*A*B + beta*C (``tsmm.execute``);
* ``grouped``  ``count`` uneven regime (i) problems in one ``tsmm.execute_grouped`` call;
* ``serve``    ``count`` requests submitted to a running ``tsmm.Server`` and drained.

``pad`` is lda - m: a column-major A straight out of a user's program has lda = m, so three quarters of
random m give an A whose columns are not 16-byte aligned.  ``dist`` names the entries of A and B:
``uniform`` in [-1, 1), or ``rows``, normal entries with every row scaled by 10**U[-3, 3].
"""
import math
import random

import torch

import paper_2208_08088_gb300 as tsmm

_DTYPES = {"f32": torch.float32, "f64": torch.float64}
_PRECISIONS = {"native": tsmm.PREC_NATIVE, "bf16x3": tsmm.PREC_BF16X3}


def _case(name, m, n, k, dtype="f32", alpha=1.0, beta=0.0, pad=0, precision="native", dist="uniform"):
    return {"name": name, "path": "execute", "dtype": dtype, "precision": precision, "m": m, "n": n, "k": k,
            "alpha": alpha, "beta": beta, "pad": pad, "dist": dist}


def _mix(name, path, count, mix, m_hi, k_hi, n_lo, n_hi):
    """``mix`` seeds the shapes: m, k and n log-uniform in [1024, m_hi], [64, k_hi] and [n_lo, n_hi]."""
    return {"name": name, "path": path, "dtype": "f32", "count": count, "mix": mix, "m_hi": m_hi, "k_hi": k_hi,
            "n_lo": n_lo, "n_hi": n_hi}


def listed():
    return [
        # one small product inside a larger program: launch and latency decide
        _case("f32_small", 2048, 16, 2048, alpha=1.5, beta=0.5),
        # the memory-bound sweep m = k = 32768: one vector, a block of 16 (accumulated into C), the widest B
        _case("f32_n1", 32768, 1, 32768),
        _case("f32_n16", 32768, 16, 32768, beta=1.0),
        _case("f32_n64", 32768, 64, 32768),
        # a typical request of the serving mix on its own: ragged sizes, columns of A not 16-byte aligned
        _case("f32_ragged", 141591, 39, 1607, alpha=1.5, beta=1.0),
        # double precision: a few right-hand sides, and the widest
        _case("f64_n4", 32768, 4, 32768, dtype="f64"),
        _case("f64_n64", 32768, 64, 32768, dtype="f64", beta=1.0),
        # rank-k updates C += A*B of a large C: thin, deep, and in double precision
        _case("rankk_f32_k16", 16384, 16384, 16, beta=1.0),
        _case("rankk_f32_k128", 16384, 16384, 128, beta=1.0),
        _case("rankk_f64_k32", 16384, 16384, 32, dtype="f64", beta=1.0),
        # the split-precision mode on entries of very different rows
        _case("bf16x3_n64", 32768, 64, 32768, precision="bf16x3", dist="rows"),
        # a burst of requests of all shapes to the server
        _mix("serve", "serve", 200, 7, 262144, 8192, 1, 64),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["tall", "tall", "tall", "tall", "tall64", "tall64", "rankk", "rankk", "rankk64", "x3", "grouped",
                       "serve"])
    alpha, beta = rng.choice([(1.0, 0.0), (1.0, 1.0), (1.5, 0.5), (-0.75, 0.0)])
    if kind == "grouped":
        n_lo = rng.choice([1, 8, 17, 33])
        c = _mix("", kind, rng.randint(12, 40), rng.randrange(1 << 20), rng.choice([8192, 65536, 262144]), 8192, n_lo,
                 min(64, 2 * n_lo))
    elif kind == "serve":
        c = _mix("", kind, rng.randint(100, 300), rng.randrange(1 << 20), 262144, 8192, 1, 64)
    else:
        f64 = kind.endswith("64")
        x3 = kind == "x3"
        tall = kind.startswith("tall") or (x3 and rng.random() < 0.5)
        while True:
            if tall:
                m, k, n = _log_int(rng, 1024, 262144), _log_int(rng, 64, 32768), _log_int(rng, 1, 64)
                size = m * k
            else:
                m, n, k = _log_int(rng, 1024, 32768), _log_int(rng, 1024, 32768), _log_int(rng, 4, 128)
                size = 4 * m * n
            if 1 << 18 <= size <= 1 << 30:  # at most the sweep's A, or the 16384 x 16384 C
                break
        if rng.random() < 0.4:  # a caller who rounds sizes
            m = m // 64 * 64
        pad = rng.choice([0, 0, 0, -m % 4, 1])
        c = _case("", m, n, k, "f64" if f64 else "f32", alpha, beta, pad, "bf16x3" if x3 else "native",
                  "rows" if rng.random() < 0.25 else "uniform")
    del c["name"]
    return c


def _shapes(case):
    """The problems (packed B's index, m, n, k, alpha, beta) of a mix and the (k, n) of its packed Bs."""
    rng = random.Random(case["mix"])
    kn = lambda: (_log_int(rng, 64, case["k_hi"]), _log_int(rng, case["n_lo"], case["n_hi"]))  # noqa: E731
    bs = [kn() for _ in range(32 if case["path"] == "serve" else case["count"])]
    probs = []
    for i in range(case["count"]):
        b = rng.randrange(len(bs)) if case["path"] == "serve" else i
        k, n = bs[b]
        m = _log_int(rng, 1024, case["m_hi"])
        probs.append((b, m, n, k, 1.0, 1.0 if i % 3 == 2 else 0.0))  # every third accumulates into C
    return bs, probs


def _fill(rows, cols, dtype, dist, gen, ld=None):
    """A rows x cols column-major matrix."""
    M = tsmm.colmajor(rows, cols, dtype, ld=ld)
    buf = M.t()._base if M.t()._base is not None else M.t()
    if dist == "uniform":
        buf.uniform_(-1.0, 1.0, generator=gen)
    else:
        buf.normal_(generator=gen)
        scale = torch.empty(rows, dtype=dtype, device="cuda").uniform_(-3.0, 3.0, generator=gen)
        M.mul_(torch.pow(10.0, scale)[:, None])
    return M


def _pool(case, gen):
    """Inputs of a mix: the Bs, one read-only pool whose windows are the As, and one buffer that holds the Cs."""
    bs, probs = _shapes(case)
    rng = random.Random(case["mix"] + 1)
    B = [_fill(k, n, torch.float32, "uniform", gen) for k, n in bs]
    pool = torch.empty(max(m * k for _, m, _, k, _, _ in probs) + 4096, dtype=torch.float32, device="cuda")
    pool.uniform_(-1.0, 1.0, generator=gen)
    total = sum(-(-m * n // 64) * 64 for _, m, n, _, _, _ in probs)
    Cs = torch.empty(total, dtype=torch.float32, device="cuda").uniform_(-1.0, 1.0, generator=gen)
    A, C, at = [], [], 0
    for _, m, n, k, _, _ in probs:
        off = rng.randrange((pool.numel() - m * k) // 64 + 1) * 64
        A.append(pool[off:off + m * k].view(k, m).t())
        C.append(Cs[at:at + m * n].view(n, m).t())
        at += -(-m * n // 64) * 64
    return B, probs, A, C, Cs


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    if case["path"] == "execute":
        dt, m, n, k = _DTYPES[case["dtype"]], case["m"], case["n"], case["k"]
        precision = _PRECISIONS[case["precision"]]
        A = _fill(m, k, dt, case["dist"], gen, m + case["pad"])
        B = _fill(k, n, dt, case["dist"], gen)
        C = _fill(m, n, dt, "uniform", gen)
        return {"path": "execute", "A": A, "C": C, "alpha": case["alpha"], "beta": case["beta"],
                "pb": tsmm.pack_b(B, precision=precision), "plan": tsmm.plan(m, n, k, dt, precision)}
    B, probs, A, C, Cs = _pool(case, gen)
    pb = [tsmm.pack_b(b) for b in B]
    if case["path"] == "grouped":
        items = [(tsmm.plan(m, n, k, tsmm.F32), alpha, A[i], pb[b], beta, C[i])
                 for i, (b, m, n, k, alpha, beta) in enumerate(probs)]
        return {"path": "grouped", "items": items, "Cs": Cs}
    torch.cuda.synchronize()  # the server's streams are not ordered after this one
    requests = [(i, pb[b], m, alpha, A[i], beta, C[i], 0.0) for i, (b, m, n, k, alpha, beta) in enumerate(probs)]
    return {"path": "serve", "server": tsmm.Server(40 << 30), "requests": requests, "Cs": Cs, "pb": pb}


def run(state):
    if state["path"] == "execute":
        tsmm.execute(state["plan"], state["alpha"], state["A"], state["pb"], state["beta"], state["C"])
        return state["C"]
    if state["path"] == "grouped":
        tsmm.execute_grouped(state["items"])
        return state["Cs"]
    state["server"].submit(state["requests"])
    state["server"].drain()
    state["server"].poll(len(state["requests"]))
    return state["Cs"]


def exact(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)

    def product(A, B, C, alpha, beta):
        P = torch.empty(C.shape[1], C.shape[0], dtype=torch.float64, device="cuda").t()
        step = max(1, (1 << 30) // max(A.shape[1], C.shape[1], 1))
        Bd = B.double()
        for i in range(0, A.shape[0], step):
            P[i:i + step] = (A[i:i + step].double() @ Bd).mul_(alpha)
        return P.add_(C.double(), alpha=beta) if beta else P

    if case["path"] == "execute":
        dt, m, n, k = _DTYPES[case["dtype"]], case["m"], case["n"], case["k"]
        A = _fill(m, k, dt, case["dist"], gen, m + case["pad"])
        B = _fill(k, n, dt, case["dist"], gen)
        C = _fill(m, n, dt, "uniform", gen)
        return product(A, B, C, case["alpha"], case["beta"])
    B, probs, A, C, Cs = _pool(case, gen)
    out, at = Cs.double(), 0
    for i, (b, m, n, _, alpha, beta) in enumerate(probs):
        out[at:at + m * n].view(n, m).t().copy_(product(A[i], B[b], C[i], alpha, beta))
        at += -(-m * n // 64) * 64
    return out


def work(case):
    """Each operand read once and C written once; 2*m*n*k operations a product."""
    es = 8 if case["dtype"] == "f64" else 4
    probs = [(0, case["m"], case["n"], case["k"], case["alpha"], case["beta"])] if case["path"] == "execute" \
        else _shapes(case)[1]
    read, flops, seen = 0, 0, set()
    for b, m, n, k, _, beta in probs:
        read += es * (m * k + m * n * (2 if beta else 1) + (0 if b in seen else k * n))
        flops += 2 * m * n * k
        seen.add(b)
    return {"bytes": read, "flops": flops}
