"""What a user of this package has it do, as timed cases.

A program that trains with GreedyLore keeps one handle per layer matrix (``GreedyLore``) and calls
``step`` or ``glr_step_group`` with every iteration's node gradients; each period opens with a
Semi-Lazy SVD refresh.  So a case is one such call, or the few calls that belong together:

* ``step``     one compressed step, somewhere inside a period (error feedback live, moments warm);
* ``refresh``  a forced refresh step, followed under Algorithm 3 (whose refresh step uses the
               uncompressed mean) by the first compressed step on the new basis;
* ``period``   one whole period of the schedule, refresh included.

The stacks are the repository's own workloads: one small fp32 matrix, the ResNet-style stack of
conv gradients (fp32, truncated and paper-exact full basis), LLaMA-style decoder layers (bf16
gradients, Adam) and the refresh-stress matrix, and fp32 matrices of ragged sizes in both
orientations.  Gradients are G_i = A diag(s) B^T + c N(0, 1) / sqrt(n) with orthonormal A, B.

The weights start at zero, so that the returned weights are the sum of the updates.
"""
import math

import torch

import paper_2507_08784_gb300 as glr

FAR = 1 << 30          # a period that no timing run reaches: refreshes are asked for, not scheduled


def _case(name, do, stack, nodes, rank, basis, dtype, opt, alg, decay, rate, rho, noise, **size):
    c = dict(do=do, stack=stack, nodes=nodes, rank=rank, basis=basis, dtype=dtype, opt=opt, alg=alg, decay=decay,
             rate=rate, rho=rho, noise=noise, **size)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest use: one 256 x 128 matrix, a whole period of five single-matrix steps (latency and launches)
        _case("matrix-period", "period", "one", 4, 4, 0, "f32", "msgd", "alg3", "power", 1.0, 16, 0.05, m=256, n=128,
              tau=5),
        # CIFAR-style pre-training: every conv layer of a ResNet-18-like stack in one grouped call
        _case("conv-step", "step", "conv", 8, 8, 16, "f32", "msgd", "alg3", "power", 1.5, 64, 0.02, width=64, levels=4),
        # ... the start of a period there
        _case("conv-refresh", "refresh", "conv", 8, 8, 16, "f32", "msgd", "alg3", "power", 1.5, 64, 0.02, width=64,
              levels=4),
        # ... and both with the full singular basis, as the paper states the method
        _case("conv-exact-step", "step", "conv", 8, 8, 0, "f32", "msgd", "alg3", "power", 1.5, 64, 0.02, width=64,
              levels=4),
        _case("conv-exact-refresh", "refresh", "conv", 8, 8, 0, "f32", "msgd", "alg3", "power", 1.5, 64, 0.02,
              width=64, levels=4),
        # layers whose sizes fit no tile (classifier heads, small embeddings), both orientations, Adam
        _case("ragged-step", "step", "ragged", 3, 5, 24, "f32", "adam", "alg3", "power", 1.0, 48, 0.03, m=333, n=777,
              count=4),
        # language-model pre-training with many nodes and a small rank: two d = 2048 decoder layers
        _case("decoder2048-step", "step", "decoder", 8, 32, 64, "bf16", "adam", "alg3", "power", 1.0, 256, 0.01,
              d=2048, ffn=5632, layers=2),
        # ... with the large rank of the d = 4096 model: two decoder layers
        _case("decoder4096-step", "step", "decoder", 4, 128, 256, "bf16", "adam", "alg3", "power", 1.2, 512, 0.01,
              d=4096, ffn=11008, layers=2),
        # ... the refresh of one d = 4096 layer's seven matrices
        _case("decoder4096-refresh", "refresh", "decoder", 4, 128, 256, "bf16", "adam", "alg4", "exp", 40.0, 512, 0.01,
              d=4096, ffn=11008, layers=1),
        # the refresh-stress matrix: a refresh in every step
        _case("stress-refresh", "refresh", "one", 8, 128, 128, "bf16", "msgd", "alg4", "exp", 40.0, 512, 0.01, m=4096,
              n=11008),
        # the paper-exact basis at decoder size: one layer's step, and one matrix's refresh
        _case("decoder2048-exact-step", "step", "decoder", 8, 32, 0, "bf16", "adam", "alg3", "power", 1.0, 256, 0.01,
              d=2048, ffn=5632, layers=1),
        _case("matrix2048-exact-refresh", "refresh", "one", 4, 32, 0, "bf16", "msgd", "alg4", "exp", 20.0, 256, 0.01,
              m=2048, n=2048),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["one", "conv", "conv", "conv-exact", "ragged", "decoder", "decoder", "decoder-refresh",
                       "stress", "exact"])
    if kind == "one":
        m, n = _log(rng, 32, 256), _log(rng, 64, 512)
        return _case(None, "period", "one", rng.randint(1, 8), rng.randint(1, 8), 0, "f32", "msgd", "alg3", "power",
                     1.0, 16, 0.05, m=m, n=n, tau=rng.randint(3, 8))
    if kind in ("conv", "conv-exact"):
        do = rng.choice(["step", "refresh"])
        basis = 0 if kind == "conv-exact" else rng.choice([16, 20, 24, 32])
        return _case(None, do, "conv", rng.randint(2, 8), rng.randint(2, 12), basis, "f32",
                     rng.choice(["msgd", "adam"]), "alg3", "power", 1.5, 64, 0.02, width=rng.randint(33, 64),
                     levels=rng.randint(2, 4))
    if kind == "ragged":
        return _case(None, "step", "ragged", rng.randint(1, 6), rng.randint(2, 12), rng.choice([16, 24, 31]), "f32",
                     rng.choice(["msgd", "adam", "adamw"]), "alg3", "power", 1.0, 48, 0.03, m=_log(rng, 64, 640),
                     n=_log(rng, 400, 1600), count=rng.randint(1, 6))
    if kind == "decoder":
        d = 8 * _log(rng, 64, 512)
        rank = 4 * rng.randint(4, 32)
        return _case(None, "step", "decoder", rng.randint(2, 8), rank, min(256, rank + 4 * rng.randint(8, 32)), "bf16",
                     "adam", "alg3", "power", rng.choice([1.0, 1.2]), 256, 0.01, d=d, ffn=8 * ((d * 11) // 32), layers=1)
    if kind == "decoder-refresh":
        d = 8 * _log(rng, 96, 512)
        rank = 4 * rng.randint(4, 32)
        return _case(None, "refresh", "decoder", rng.randint(2, 4), rank, min(256, 2 * rank), "bf16", "adam", "alg4",
                     "exp", max(8.0, rank / 3.2), 512, 0.01, d=d, ffn=8 * ((d * 11) // 32), layers=1)
    if kind == "stress":
        m, n = 8 * _log(rng, 128, 512), 8 * _log(rng, 256, 1376)
        rank = 4 * rng.randint(8, 32)
        return _case(None, "refresh", "one", rng.randint(2, 8), rank, rank, "bf16", "msgd", "alg4", "exp",
                     max(8.0, rank / 3.2), 512, 0.01, m=m, n=n)
    m = 128 * rng.randint(9, 16)
    n = m + 8 * rng.randint(0, 128)
    do = rng.choice(["step", "refresh"])
    if do == "step":
        return _case(None, "step", "one", rng.randint(2, 8), 4 * rng.randint(4, 16), 0, "bf16", "adam", "alg3", "power",
                     1.0, 256, 0.01, m=m, n=n)
    rank = 4 * rng.randint(4, 16)
    return _case(None, "refresh", "one", rng.randint(2, 8), rank, 0, "bf16", "msgd", "alg4", "exp",
                 max(8.0, rank / 1.6), 256, 0.01, m=m, n=n)


def _shapes(c):
    """(m, n) of every matrix of the case, as its gradient is laid out."""
    if c["stack"] == "one":
        return [(c["m"], c["n"])]
    if c["stack"] == "conv":           # out_ch x (in_ch * 9), two of each level
        return [(c["width"] << l, (c["width"] << l) * 9) for l in range(c["levels"]) for _ in range(2)]
    if c["stack"] == "ragged":         # sizes that shrink by odd amounts, every second one transposed
        out = []
        for i in range(c["count"]):
            m, n = max(48, c["m"] - 37 * i), max(64, c["n"] - 91 * i)
            out.append((n, m) if i % 2 else (m, n))
        return out
    d, f = c["d"], c["ffn"]
    return ([(d, d)] * 4 + [(f, d)] * 2 + [(d, f)]) * c["layers"]


def _sizes(c, shape):
    mp, np_ = min(shape), max(shape)
    r = min(c["rank"], mp)
    k = mp if c["basis"] == 0 else min(c["basis"], mp)
    return mp, np_, r, max(k, r)


def _spectrum(c, rho, device="cuda"):
    j = torch.arange(1, rho + 1, dtype=torch.float64, device=device)
    return j ** -c["rate"] if c["decay"] == "power" else torch.exp(-j / c["rate"])


def _generator(seed, *tag):
    g = torch.Generator(device="cuda")
    s = seed & 0x7FFFFFFF
    for t in tag:
        s = (s * 1_000_003 + t + 1) & 0x7FFFFFFFFFFF
    g.manual_seed(s)
    return g


class _Frames:
    """Orthonormal columns per dimension, drawn once; a matrix takes a row permutation with signs of it."""

    def __init__(self, c, seed):
        self.c, self.seed, self.base, self.cols = c, seed, {}, {}
        for shape in _shapes(c):
            mp, np_, _, k = _sizes(c, shape)
            for dim, want in ((mp, max(min(c["rho"], mp), k)), (np_, min(c["rho"], mp))):
                self.cols[dim] = min(dim, max(self.cols.get(dim, 0), want))

    def frame(self, dim, tag):
        if dim not in self.base:
            x = torch.randn(dim, self.cols[dim], dtype=torch.float64, device="cuda",
                            generator=_generator(self.seed, 1, dim))
            self.base[dim] = torch.linalg.qr(x)[0]
        g = _generator(self.seed, 2, dim, tag)
        perm = torch.randperm(dim, device="cuda", generator=g)
        sign = torch.randint(0, 2, (dim, 1), device="cuda", generator=g).double() * 2 - 1
        return self.base[dim][perm] * sign


def _program(c):
    """What is called: lists of (refresh asked for, gradient set) before and in the timed pass, the
    gradient sets, the warm-up steps, and after which prepared step the basis is set (-1: before all)."""
    if c["do"] == "period":
        return [], [(False, i) for i in range(c["tau"])], c["tau"], 0, None
    if c["do"] == "step":       # warm-up, the refresh, one compressed step; then another compressed step
        return [(False, 0), (True, 1), (False, 0)], [(False, 1)], 2, 1, 1
    steps = [(True, 0)] if c["alg"] == "alg4" else [(True, 0), (False, 1)]
    return [(False, 0), (False, 1)], steps, 2, 2, -1


def _matrix(c, frames, seed, i, shape):
    """Matrix i's gradients, [set][node], and its basis (the last period's: the leading left vectors,
    disturbed a little where a refresh starts from it)."""
    mp, np_, r, k = _sizes(c, shape)
    rho = min(c["rho"], mp)
    A, B = frames.frame(mp, 2 * i), frames.frame(np_, 2 * i + 1)
    S = ((A[:, :rho] * _spectrum(c, rho)).float() @ B[:, :rho].float().T)
    if shape[0] > shape[1]:
        S = S.T
    dt = torch.float32 if c["dtype"] == "f32" else torch.bfloat16
    scale = c["noise"] / math.sqrt(shape[1])
    g = _generator(seed, 3, i)
    G = [[torch.add(S, torch.randn(shape, device="cuda", generator=g), alpha=scale).to(dt).contiguous()
          for _ in range(c["nodes"])] for _ in range(_program(c)[2])]
    Q = A[:, :k]
    if c["do"] == "refresh":
        if k < mp:
            Q = torch.linalg.qr(Q + 0.05 * torch.randn(mp, k, dtype=torch.float64, device="cuda", generator=g)
                                / math.sqrt(mp))[0]
    return G, Q.float().contiguous()


_OPT = {"msgd": dict(optimizer="msgd", lr=0.01, beta1=0.9),
        "adam": dict(optimizer="adam", lr=1e-3, beta1=0.9, beta2=0.999, eps=1e-8),
        "adamw": dict(optimizer="adamw", lr=1e-3, beta1=0.9, beta2=0.999, eps=1e-8, weight_decay=0.01)}


def _vseed(seed, i):
    return (seed * 7919 + 104729 * i + 17) & 0x7FFFFFFF


class _State:
    pass


def prepare(case, seed):
    before, steps, _, warm, basis_at = _program(case)
    s = _State()
    s.steps, s.alone = steps, case["stack"] == "one"
    s.handles, s.X, s.G = [], [], []
    frames = _Frames(case, seed)
    bases = []
    for i, shape in enumerate(_shapes(case)):
        mp, np_, r, k = _sizes(case, shape)
        G, Q = _matrix(case, frames, seed, i, shape)
        s.handles.append(glr.GreedyLore(shape[0], shape[1], r, case["nodes"], tau=case.get("tau", FAR),
                                        refresh_mode=case["alg"], seed=_vseed(seed, i),
                                        basis_rank=0 if k == mp else k, power_iters=4, grad_dtype=case["dtype"],
                                        compress_start=warm, **_OPT[case["opt"]]))
        s.X.append(torch.zeros(shape, device="cuda"))
        s.G.append(G)
        bases.append(Q)
    del frames

    def set_bases():
        for h, Q in zip(s.handles, bases):
            h.set_basis(Q)

    if basis_at == -1:
        set_bases()
    for j, (refresh, which) in enumerate(before):
        _one(s, refresh, which)
        if basis_at == j:
            set_bases()
    torch.cuda.synchronize()
    return s


def _one(s, refresh, which):
    if refresh:
        for h in s.handles:
            h.refresh()
    if s.alone:
        s.handles[0].step(s.G[0][which], s.X[0])
    else:
        glr.glr_step_group(s.handles, [g[which] for g in s.G], s.X)


def run(state):
    for refresh, which in state.steps:
        _one(state, refresh, which)
    return state.X


def work(case):
    """Each gradient, error and weight read once, errors and weights written once; the rank-r products of
    error feedback, the scores' and the refresh's products."""
    gs = 4 if case["dtype"] == "f32" else 2
    opt = 16 if case["opt"] == "msgd" else 24
    q = 4
    b = f = 0.0
    _, steps, _, _, _ = _program(case)
    for shape in _shapes(case):
        mp, np_, r, k = _sizes(case, shape)
        e, N = float(mp) * np_, case["nodes"]
        full = k == mp
        for j, (refresh, _) in enumerate(steps):
            refresh = refresh or (case["do"] == "period" and j == 0)
            compressed = not refresh or case["alg"] == "alg4"
            b += N * e * (gs + 4 + (4 if compressed else 0)) + e * opt
            f += 4 * N * e * r + (2 * e * r if compressed else 0)
            if refresh:
                f += (2 * e * mp + 9 * float(mp) ** 3) if full else (2 * q + 1) * 2 * e * k
            else:
                f += 2 * e * mp if full else 4 * e * k
    return {"bytes": b, "flops": f}


def tolerance(case):
    """About four times what the start of this file's use showed against exact(): 7e-6 at most for fp32
    gradients (Adam's beta2 in fp32), 7e-4 for the TF32 refreshes.  A bf16 step is off by as little unless
    two scores of the selection lie within their TF32 rounding, which swaps a column of P: 3e-3 to 3e-2."""
    if case["dtype"] == "f32":
        return {"rel": 3e-5, "max": 1e-2}
    return {"rel": 3e-3, "max": 0.3} if case["do"] == "refresh" else {"rel": 2e-2, "max": 0.8}


# ---- the same in 64 bits, from the method's definition ------------------------------------------

def _philox(c, k0, k1):
    """Philox4x32-10 (Salmon et al., SC'11) on int64 tensors that hold 32-bit words."""
    mask = 0xFFFFFFFF
    for rnd in range(10):
        p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57
        hi0, lo0 = (p0 >> 32) & mask, p0 & mask
        hi1, lo1 = (p1 >> 32) & mask, p1 & mask
        c = [hi1 ^ c[1] ^ k0, lo1, hi0 ^ c[3] ^ k1, lo0]
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    return c


def _vectors(seed, t, rows, cols):
    """The shared random vectors v_j of step t, one a row: Box-Muller on the words of counter (b / 4, j, t, tag)."""
    nq = (cols + 3) // 4
    j = torch.arange(rows, device="cuda").view(-1, 1).expand(rows, nq)
    b = torch.arange(nq, device="cuda").view(1, -1).expand(rows, nq)
    w = _philox([b, j, torch.full_like(j, t), torch.full_like(j, 0x4C414D56)], seed & 0xFFFFFFFF, seed >> 32)
    u = [((x >> 9).double() + 0.5) * 2.0 ** -23 for x in w]
    out = torch.empty(rows, nq, 4, dtype=torch.float64, device="cuda")
    for q in (0, 2):
        rad = torch.sqrt(-2.0 * torch.log(u[q]))
        out[:, :, q] = rad * torch.cos(2 * math.pi * u[q + 1])
        out[:, :, q + 1] = rad * torch.sin(2 * math.pi * u[q + 1])
    return out.view(rows, nq * 4)[:, :cols]


def _complete(Q):
    """[Q, the rest of an orthogonal matrix by Householder's QR of Q]."""
    if Q.shape[0] == Q.shape[1]:
        return Q
    U = torch.linalg.qr(Q, mode="complete")[0].clone()
    U[:, :Q.shape[1]] = Q
    return U


def _new_basis(Mbar, Q, k):
    """The refresh: the singular basis of the mean, or its leading part by four block power iterations
    from Q with a Rayleigh-Ritz step."""
    if k == Mbar.shape[0]:
        return torch.linalg.eigh(Mbar @ Mbar.T)[1].flip(1)
    for _ in range(4):
        Z = torch.linalg.qr(Mbar.T @ Q)[0]
        Q = torch.linalg.qr(Mbar @ Z)[0]
    Z = Mbar.T @ Q
    return _complete(Q @ torch.linalg.eigh(Z.T @ Z)[1].flip(1))


def exact(case, seed):
    before, steps, _, warm, basis_at = _program(case)
    opt, out = _OPT[case["opt"]], []
    frames = _Frames(case, seed)
    for i, shape in enumerate(_shapes(case)):
        mp, np_, r, k = _sizes(case, shape)
        flip = shape[0] > shape[1]
        G, Q0 = _matrix(case, frames, seed, i, shape)
        Q0 = Q0.double()
        X, Mo, Vo = (torch.zeros(shape, dtype=torch.float64, device="cuda") for _ in range(3))
        E, U, Q = None, None, Q0
        if basis_at == -1:
            U = _complete(Q0)
        for t, (asked, which) in enumerate(before + steps):
            M = [(g.T if flip else g).double() for g in G[which]]
            if t >= warm and E is not None:
                M = [a + e for a, e in zip(M, E)]
            Mbar = sum(M) / len(M)
            refresh = t >= warm and (asked or t == warm or (t - warm) % case.get("tau", FAR) == 0)
            if t < warm:
                D = Mbar
            else:
                if refresh:
                    U = _new_basis(Mbar, Q, k) if not (basis_at == t) else None
                    Q = None if U is None else U[:, :k]
                if refresh and case["alg"] == "alg3":
                    E, D = None, Mbar
                else:
                    if refresh:
                        J = torch.arange(r, device="cuda")
                    else:
                        lam = ((U.T @ Mbar) * _vectors(_vseed(seed, i), t, mp, np_)).sum(1)
                        J = torch.topk(lam * lam, r)[1]
                    P = U[:, J]
                    E = [a - P @ (P.T @ a) for a in M]
                    D = P @ (P.T @ Mbar)
            if flip:
                D = D.T
            Mo = opt["beta1"] * Mo + (1 - opt["beta1"]) * D
            if case["opt"] == "msgd":
                X = X - opt["lr"] * Mo
            else:
                Vo = opt["beta2"] * Vo + (1 - opt["beta2"]) * D * D
                a, b = Mo, Vo
                if case["opt"] == "adamw":
                    a, b = Mo / (1 - opt["beta1"] ** (t + 1)), Vo / (1 - opt["beta2"] ** (t + 1))
                X = X - opt["lr"] * (a / (torch.sqrt(b) + opt["eps"]) + opt.get("weight_decay", 0.0) * X)
            if basis_at == t:
                U, Q = _complete(Q0), Q0
        out.append(X)
        del G, M, E, U, Mo, Vo
    return out
