"""The measured workloads of the multi-scale low rank decomposition library.

Each case is one call a user's program makes through the Python binding of
the C ABI: a single block singular value threshold (msllr_blocksvt, eq:bsvt
under a cycle-spin shift) or a whole decomposition (msllr_decompose on device
buffers, msllr_decompose_host on pinned host buffers, msllr_decompose_batch
over stacked jobs).  Sizes come from the benchmark's workloads (64 x 64,
16384 x 256 video, 512/1024 jobs, ratings, 8192 x 8192) or are drawn from the
ranges between them.

Inputs follow the seeded generators of synth.py (block-wise low rank terms
per scale, sparse entries, dense noise), drawn on the GPU.
"""

import math

import numpy as np
import torch

from paper_1507_08751_gb300 import binding as B

DEV = "cuda"


# ---------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------
def _svt(name, M, N, m, n, ranks, noise):
    """One block SVT: blocks hold up to `ranks` terms over dense noise."""
    c = {"kind": "svt", "M": M, "N": N, "m": m, "n": n, "ranks": ranks, "noise": noise}
    if name:
        c["name"] = name
    return c


def _admm(name, entry, M, N, scales, iters, data, batch=1, mask=False, area=False):
    """One decomposition; `scales` as text "m x n,..." (plain values only)."""
    c = {"kind": "admm", "entry": entry, "M": M, "N": N, "iters": iters, "batch": batch,
         "scales": ",".join("%dx%d" % s for s in scales), "data": data, "mask": mask, "area": area}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call: one prox of a 64 x 64 matrix by 16 x 16 blocks;
        # launches, the call's synchronisation and copies are what counts
        _svt("svt_64x64_by16", 64, 64, 16, 16, 1, 0.5),
        # the narrow scales of the video matrix, one prox each: thousands of
        # blocks, most of them of rank 0
        _svt("svt_video_by16", 16384, 256, 16, 16, 1, 0.5),
        _svt("svt_video_by64", 16384, 256, 64, 64, 2, 0.6),
        # the 256-wide scale of the video matrix: few terms per block
        _svt("svt_video_by256", 16384, 256, 256, 256, 3, 0.6),
        # 256-wide blocks as a settled job holds them: up to 12 terms a block
        _svt("svt_1024_by256_rank12", 1024, 1024, 256, 256, 12, 0.6),
        # plain SVT of a 1024 x 1024 matrix (the full-matrix scale of a job)
        _svt("svt_1024_full", 1024, 1024, 1024, 1024, 6, 0.3),
        # the smallest decomposition, launch and latency bound throughout
        _admm("admm_64", "device", 64, 64, [(1, 1), (4, 4), (16, 16), (64, 64)], 30, "blocks",
              area=True),
        # the flagship: the surveillance-video shape with its five scales
        _admm("admm_video", "device", 16384, 256,
              [(1, 1), (16, 16), (64, 64), (256, 256), (16384, 256)], 30, "blocks"),
        # a batching/serving job of six dyadic scales with a 1024-wide one
        _admm("admm_job1024", "device", 1024, 1024,
              [(1, 1), (4, 4), (16, 16), (64, 64), (256, 256), (1024, 1024)], 8, "blocks"),
        # sixteen jobs of one shape in shared launches
        _admm("admm_batch16_512", "batch", 512, 512,
              [(1, 1), (4, 4), (16, 16), (64, 64), (512, 512)], 10, "blocks", batch=16),
        # a user x item rating matrix with its mask, from and to host memory:
        # sizes that are no powers of two, wide (transposed) blocks
        _admm("host_ratings_4080x510", "host", 4080, 510,
              [(1, 1), (5, 5), (15, 15), (51, 85), (102, 170), (4080, 510)], 8, "ratings",
              mask=True),
        # the largest: the 8192 x 8192 matrix with blocks up to its full width
        _admm("admm_8192", "device", 8192, 8192,
              [(1, 1), (8, 8), (32, 32), (128, 128), (1024, 1024), (8192, 8192)], 2, "spread"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    if rng.random() < 0.5:
        # one prox: blocks 2 .. 512 wide, square to 4:1 either way, and from
        # one block to as many as 4M entries hold
        w = _log_int(rng, 2, 512)
        m, n = w, w
        if rng.random() < 0.5:
            o = _log_int(rng, w, 4 * w)
            m, n = (o, w) if rng.random() < 0.7 else (w, o)
        room = max(1, (1 << 22) // (m * n))
        nb = _log_int(rng, 1, min(room, 4096))
        bn = _log_int(rng, 1, nb)
        bm = max(1, nb // bn)
        return _svt(None, m * bm, n * bn, m, n, rng.randint(1, 12 if w > 64 else 3),
                    round(rng.uniform(0.3, 0.7), 3))
    # a decomposition: 1 x 1, two to four dyadic block sizes and the full
    # matrix, sides odd multiples of the widest block
    base = rng.choice((2, 3, 4, 4, 5))
    sizes, b = [], base
    while b <= 256 and len(sizes) < 4:
        if b >= 4:
            sizes.append(b)
        b *= base
    sizes = sizes[:rng.randint(2, len(sizes))]
    big = sizes[-1]
    N = big * max(1, _log_int(rng, 64, 1024) // big)
    M = big * max(1, _log_int(rng, N, max(2 * N, min(8192, (1 << 21) // N))) // big)
    scales = [(1, 1)] + [(s, s) for s in sizes] + ([(M, N)] if (M, N) != (big, big) else [])
    entry = rng.choice(("device", "device", "host", "batch"))
    batch = rng.randint(2, 8) if entry == "batch" and M * N <= (1 << 18) else 1
    if batch == 1 and entry == "batch":
        entry = "device"
    ratings = rng.random() < 0.3
    return _admm(None, entry, M, N, scales, rng.randint(2, 8), "ratings" if ratings else "blocks",
                 batch=batch, mask=ratings)


def _scales(case):
    return [tuple(int(v) for v in s.split("x")) for s in case["scales"].split(",")]


def _lambdas(case):
    M, N = case["M"], case["N"]
    if case["area"]:
        return [math.sqrt(m) + math.sqrt(n) + math.sqrt(math.log(M * N / (m * n)))
                for m, n in _scales(case)]
    return [math.sqrt(m) + math.sqrt(n) + math.sqrt(math.log(M * N / max(m, n)))
            for m, n in _scales(case)]


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def _terms(g, M, N, m, n, rank, p, amp=None):
    """Each m x n block active with probability p, then a sum of up to `rank`
    Gaussian outer products; amp = (lo, hi): unit vectors with singular values
    log-uniform between them instead."""
    bm, bn = M // m, N // n
    u = torch.randn((bm, bn, m, rank), generator=g, device=DEV)
    v = torch.randn((bm, bn, n, rank), generator=g, device=DEV)
    on = (torch.rand((bm, bn, 1, 1), generator=g, device=DEV) < p).float()
    count = torch.randint(1, rank + 1, (bm, bn, 1, 1), generator=g, device=DEV)
    on = on * (torch.arange(rank, device=DEV) < count)
    if amp is not None:
        u = u / u.norm(dim=2, keepdim=True).clamp_min(1e-20)
        v = v / v.norm(dim=2, keepdim=True).clamp_min(1e-20)
        lo, hi = math.log(amp[0]), math.log(amp[1])
        on = on * torch.exp(lo + (hi - lo) * torch.rand((bm, bn, 1, rank), generator=g, device=DEV))
    X = torch.matmul(u * on, v.transpose(2, 3))
    return X.permute(0, 2, 1, 3).reshape(M, N)


def _svt_input(case, seed):
    """A prox input on the grid moved by a random shift: dense noise whose
    singular values stay below tau, and block terms from half to six times
    tau, which the moved grid cuts into pieces around tau."""
    g = _gen(seed)
    M, N, m, n = case["M"], case["N"], case["m"], case["n"]
    tau = math.sqrt(m) + math.sqrt(n) + math.sqrt(math.log(M * N / max(m, n)))
    A = case["noise"] * torch.randn((M, N), generator=g, device=DEV)
    p = 1.0 if (M // m) * (N // n) < 32 else 0.2
    A += _terms(g, M, N, m, n, case["ranks"], p, (0.5 * tau, 6.0 * tau))
    sh = torch.randint(0, 1 << 30, (2,), generator=g, device=DEV).tolist()
    return A, tau, (sh[0] % M, sh[1] % N)


def _admm_input(case, seed):
    g = _gen(seed)
    M, N, scales = case["M"], case["N"], _scales(case)
    Ys, masks = [], []
    for _ in range(case["batch"]):
        if case["data"] == "ratings":
            # 5 % observed entries, integer values 1..5
            mask = torch.rand((M, N), generator=g, device=DEV) < 0.05
            Y = torch.randint(1, 6, (M, N), generator=g, device=DEV).float() * mask
            masks.append(mask.to(torch.uint8))
        else:
            # rank-1/2 terms in a few per cent of every scale's blocks, one
            # global term, 2 % sparse entries ("spread": singular values
            # log-uniform over [1e-2, 1e2], some near their scale's threshold)
            Y = torch.randn((M, N), generator=g, device=DEV)
            Y *= torch.rand((M, N), generator=g, device=DEV) < 0.02
            for m, n in scales[1:]:
                full = (m, n) == (M, N)
                Y += _terms(g, M, N, m, n, 2, 1.0 if full else 0.03,
                            (1e-2, 1e2) if case["data"] == "spread" else None)
        Ys.append(Y)
    return torch.stack(Ys), (torch.stack(masks) if masks else None)


_contexts = {}


def _context():
    # one context per process, as a program keeps it
    if "ctx" not in _contexts:
        _contexts["ctx"] = B.Context(0)
    return _contexts["ctx"]


def prepare(case, seed):
    st = {"case": case, "ctx": _context(), "seed": int(seed) & 0x7FFFFFFF}
    if case["kind"] == "svt":
        st["A"], st["tau"], st["shift"] = _svt_input(case, seed)
        st["Z"] = torch.empty_like(st["A"])
        return st
    Y, mask = _admm_input(case, seed)
    L, b, M, N = len(_scales(case)), case["batch"], case["M"], case["N"]
    st["scales"], st["lam"] = _scales(case), _lambdas(case)
    if case["entry"] == "batch":
        st["Y"], st["mask"] = Y, mask
        st["X"] = torch.empty((L, b, M, N), device=DEV)
        st["Z"] = torch.empty((L, b, M, N), device=DEV)
        st["seeds"] = [st["seed"] + 101 * j for j in range(b)]
        return st
    Y, mask = Y[0], None if mask is None else mask[0]
    if case["entry"] == "host":
        st["Y"] = Y.cpu().pin_memory()
        st["mask"] = None if mask is None else mask.cpu().pin_memory()
        st["X"] = torch.empty((L, M, N), pin_memory=True)
        st["Z"] = torch.empty((L, M, N), pin_memory=True)
        return st
    st["Y"], st["mask"] = Y.contiguous(), mask
    st["X"] = torch.empty((L, M, N), device=DEV)
    st["Z"] = torch.empty((L, M, N), device=DEV)
    return st


def run(st):
    case, ctx = st["case"], st["ctx"]
    if case["kind"] == "svt":
        ctx.msllr_blocksvt(st["A"], st["Z"], case["m"], case["n"], st["tau"], st["shift"])
        return st["Z"]
    if case["entry"] == "batch":
        ctx.msllr_decompose_batch(st["Y"], st["scales"], st["X"], st["seeds"], lambdas=st["lam"],
                                  iters=case["iters"], mask=st["mask"], Z_out=st["Z"])
    else:
        f = ctx.msllr_decompose_host if case["entry"] == "host" else ctx.msllr_decompose
        f(st["Y"], st["scales"], st["X"], lambdas=st["lam"], iters=case["iters"], seed=st["seed"],
          mask=st["mask"], Z_out=st["Z"])
    return {"X": st["X"], "Z": st["Z"]}


def work(case):
    """One pass.  A prox reads A and writes Z; an ADMM iteration reads Y and
    reads and writes the two state matrices of every scale.  Flops: the Gram
    product of every block (lower triangle, a multiply-add is 2)."""
    M, N = case["M"], case["N"]

    def gram(m, n):
        if m == 1 and n == 1:
            return 2.0 * M * N
        mm, nn = max(m, n), min(m, n)
        return float(M // m) * (N // n) * mm * nn * (nn + 1)

    if case["kind"] == "svt":
        return {"bytes": 8.0 * M * N, "flops": gram(case["m"], case["n"])}
    sc, k = _scales(case), case["batch"] * case["iters"]
    return {"bytes": 4.0 * M * N * (4 * len(sc) + 1) * k,
            "flops": k * sum(gram(m, n) for m, n in sc)}


# ---------------------------------------------------------------------------
# the same results in 64 bits
# ---------------------------------------------------------------------------
def _eigh(G):
    # the batched GPU solver takes small matrices, and now and then refuses
    # one with many repeated eigenvalues: LAPACK on the host then
    out = []
    for g in (G.split(4096) if G.shape[-1] <= 256 else G.split(1)):
        try:
            out.append(torch.linalg.eigh(g))
        except RuntimeError:
            w, v = np.linalg.eigh(g.cpu().numpy())
            out.append((torch.from_numpy(w).to(g), torch.from_numpy(v).to(g)))
    return torch.cat([o[0] for o in out]), torch.cat([o[1] for o in out])


def _svt64(A, m, n, tau, shift):
    M, N = A.shape
    if m == 1 and n == 1:
        return torch.sign(A) * (A.abs() - tau).clamp_min(0.0)
    full = (m, n) == (M, N)
    if not full:
        A = torch.roll(A, (-shift[0], -shift[1]), (0, 1))
    C = A.reshape(M // m, m, N // n, n).permute(0, 2, 1, 3).reshape(-1, m, n)
    if m < n:
        C = C.transpose(1, 2)
    w, V = _eigh(C.transpose(1, 2) @ C)
    s = w.clamp_min(0.0).sqrt()
    f = torch.where(s > tau, 1.0 - tau / s.clamp_min(1e-300), torch.zeros_like(s))
    Z = (C @ (V * f[:, None, :])) @ V.transpose(1, 2)
    if m < n:
        Z = Z.transpose(1, 2)
    Z = Z.reshape(M // m, N // n, m, n).permute(0, 2, 1, 3).reshape(M, N)
    return Z if full else torch.roll(Z, shift, (0, 1))


def _shifts64(seed, iters, M, N):
    """The cycle-spin shift sequence: splitmix64 of the seed."""
    out, full = [], (1 << 64) - 1
    for k in range(iters):
        z = (seed + (k + 1) * 0x9E3779B97F4A7C15) & full
        z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & full
        z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & full
        z ^= z >> 31
        out.append(((z >> 32) % M, (z & 0xFFFFFFFF) % N))
    return out


def _admm64(Y, mask, scales, lam, iters, shifts):
    Y = Y.double()
    Z = [torch.zeros_like(Y) for _ in scales]
    U = [torch.zeros_like(Y) for _ in scales]

    def resid():
        r = (Y - sum(z - u for z, u in zip(Z, U))) / len(scales)
        return r if mask is None else r * (mask != 0)

    for k in range(iters):
        r = resid()
        for i, (m, n) in enumerate(scales):
            A = Z[i] + r
            Z[i] = _svt64(A, m, n, lam[i], shifts[k])
            U[i] = A - Z[i]
    r = resid()
    return torch.stack([z - u + r for z, u in zip(Z, U)]), torch.stack(Z)


def exact(case, seed):
    if case["kind"] == "svt":
        A, tau, sh = _svt_input(case, seed)
        return _svt64(A.double(), case["m"], case["n"], float(np.float32(tau)), sh)
    # about 0.7 us per entry and iteration
    if case["M"] * case["N"] * case["batch"] * case["iters"] > 18_000_000:
        return None
    Y, mask = _admm_input(case, seed)
    s0 = int(seed) & 0x7FFFFFFF
    seeds = [s0 + 101 * j for j in range(case["batch"])]
    lam = [float(np.float32(v)) for v in _lambdas(case)]
    got = [_admm64(Y[j], None if mask is None else mask[j], _scales(case), lam, case["iters"],
                   _shifts64(seeds[j], case["iters"], case["M"], case["N"]))
           for j in range(case["batch"])]
    X, Z = (torch.stack([x[i] for x in got], dim=1) for i in (0, 1))
    if case["entry"] != "batch":
        X, Z = X[:, 0], Z[:, 0]
    return {"X": X, "Z": Z}
