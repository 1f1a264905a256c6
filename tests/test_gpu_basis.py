"""The refreshed basis and the selection at the edges of their kernels' size classes (marked gpu):
eigenvectors against their defining properties in fp64, the truncated basis against the SVD, the
arg-top-r against a stable sort."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
EPS = 2.0 ** -24


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()


def _refreshed(m, n, r, k, G, dtype, steps=1):
    """A handle after `steps` steps on the gradient G (a refresh in the first)."""
    import torch
    import paper_2507_08784_gb300 as glr
    h = glr.GreedyLore(m, n, r, 1, tau=100, optimizer="msgd", lr=0.01, beta1=0.9, seed=5, basis_rank=k,
                       grad_dtype=dtype)
    X = torch.zeros(m, n, device="cuda")
    Gd = torch.from_numpy(G).to(torch.float32 if dtype == "f32" else torch.bfloat16).cuda()
    for _ in range(steps):
        h.step([Gd], X)
    torch.cuda.synchronize()
    h.stats()
    return h


@pytest.mark.parametrize("n", [1, 2, 3, 16, 17, 33, 64, 65, 127, 128, 129, 255, 256, 257, 384, 511, 512, 513])
def test_full_basis_eigenvectors(n):
    """U of H = Mbar Mbar^T from the cluster Jacobi (V kept in the cluster up to 256, from the logged
    rotations up to 512) and the grid-wide one (513).  The solver stops at off(H) <= (4 eps sqrt(n) + 1e-7)
    ||H||, and about 10 sweeps of n - 1 rotations, each off by a few eps, add an error that grows as
    the square root of their number: 4 eps sqrt(10 n) in U and, relative to ||H||, in U^T H U."""
    G = np.random.default_rng(n).standard_normal((n, n + 4)).astype(np.float32)
    h = _refreshed(n, n + 4, 1, 0, G, "f32")
    U = h.basis().double().cpu().numpy()
    h.close()
    H = G.astype(np.float64) @ G.T.astype(np.float64)
    D = U.T @ H @ U
    rounding = 4 * EPS * np.sqrt(10 * n)
    assert np.abs(U.T @ U - np.eye(n)).max() <= 4 * EPS + rounding
    off = np.linalg.norm(D - np.diag(np.diag(D)))
    assert off <= (4 * EPS * np.sqrt(n) + 1e-7 + 2 * rounding) * np.linalg.norm(H)
    w = np.linalg.eigvalsh(H)[::-1]
    assert np.abs(np.diag(D) - w).max() <= off + 1e-6 * w[0]


def _gapped(m, n, k, seed):
    """k singular values from 1 down to 1/2, the rest at 1/100: four power iterations (two products each)
    leave (1/50)^8 of the complement."""
    rng = np.random.default_rng(seed)
    q = min(m, n)
    U = np.linalg.qr(rng.standard_normal((m, q)))[0]
    V = np.linalg.qr(rng.standard_normal((n, q)))[0]
    s = np.full(q, 0.01)
    s[:k] = np.linspace(1.0, 0.5, k)
    return ((U * s) @ V.T).astype(np.float32)


@pytest.mark.parametrize("m,n,r,k,dtype", [
    (33, 64, 1, 1, "f32"), (40, 96, 2, 2, "f32"), (65, 132, 3, 5, "f32"), (100, 64, 4, 16, "f32"),
    (65, 1024, 4, 17, "f32"), (130, 516, 8, 31, "f32"), (512, 576, 8, 32, "f32"), (600, 640, 8, 16, "f32"),
    (136, 264, 16, 16, "bf16"), (136, 520, 16, 20, "bf16"), (264, 136, 16, 32, "bf16"), (200, 328, 16, 36, "bf16"),
    (256, 4104, 16, 64, "bf16"), (192, 328, 16, 68, "bf16"), (4104, 256, 16, 128, "bf16"),
    (256, 1288, 16, 132, "bf16"), (264, 520, 16, 256, "bf16"),
])
def test_truncated_basis(m, n, r, k, dtype):
    """The refresh of every class of k (one warp's rows, the small and the blocked eigenproblem, the blocked
    factors' 32-column panels with a remainder, sliced and whole products): an orthogonal U, its first
    k columns spanning the top-k singular subspace, diagonal there.  The last product and the
    orthonormalisation are fp32-exact, so the subspace is off by a few eps sqrt(n') over the gap 1/2
    (1e-4 allowed); H comes from TF32 products on the bf16 path, 2^-11 each."""
    G = _gapped(m, n, k, seed=m + n + k)
    h = _refreshed(m, n, r, k, G, dtype)
    J, P, Rbar, lam, Mbar = h.selection()
    U = h.basis().double().cpu().numpy()
    A = Mbar.double().cpu().numpy()
    h.close()
    assert np.abs(U.T @ U - np.eye(U.shape[0])).max() <= 2e-5
    Us = np.linalg.svd(A, full_matrices=False)[0][:, :k]
    Uk = U[:, :k]
    sine = np.linalg.norm(Uk - Us @ (Us.T @ Uk), 2)
    assert sine <= 1e-4
    D = Uk.T @ A @ A.T @ Uk
    tol = 2.0 ** -10 if dtype == "bf16" else 2e-5
    assert np.abs(D - np.diag(np.diag(D))).max() <= tol * D[0, 0]
    assert np.all(np.diff(np.diag(D)) <= 2 * tol * D[0, 0])


@pytest.mark.parametrize("m,n,r,k", [(136, 520, 16, 20), (200, 328, 16, 36), (256, 1288, 16, 132)])
@pytest.mark.parametrize("scale", [1e-6, 1.0, 1e7])
def test_truncated_basis_at_any_gradient_scale(m, n, r, k, scale):
    """k no multiple of the factors' 32-column blocks: the padding must not be taken for pivots, whatever the
    size of the real ones (their mean is 6e13 for gradients of loss-scaled size).  The subspace and the
    bounds are those of test_truncated_basis, and the handle reports no failed factorisation."""
    G = (_gapped(m, n, k, seed=m + n + k) * scale).astype(np.float32)
    h = _refreshed(m, n, r, k, G, "bf16")                # its stats() raises on a numeric failure
    A = h.selection()[4].double().cpu().numpy() / scale
    U = h.basis().double().cpu().numpy()
    h.close()
    assert np.abs(U.T @ U - np.eye(U.shape[0])).max() <= 2e-5
    Us = np.linalg.svd(A, full_matrices=False)[0][:, :k]
    assert np.linalg.norm(U[:, :k] - Us @ (Us.T @ U[:, :k]), 2) <= 1e-4


@pytest.mark.parametrize("m,n,r,k,dtype", [(96, 256, 4, 16, "f32"), (130, 516, 4, 31, "f32"), (160, 320, 4, 40, "f32"),
                                           (300, 640, 4, 264, "f32"), (136, 520, 16, 20, "bf16"), (256, 520, 16, 132, "bf16")])
@pytest.mark.parametrize("scale", [2.0 ** -17, 1.0, 2.0 ** 17])
def test_rank_deficient_refresh_at_any_gradient_scale(m, n, r, k, dtype, scale):
    """Gradients of rank 4 < k: the Gram matrices are singular to rounding and every factor needs a diagonal
    shift, which has to grow from attempt to attempt relative to the matrix.  No factorisation is
    given up, and the leading four basis vectors span the gradient's column space at each scale: in fp32 to
    rounding (about 3e-7 in a CPU model of the iteration; 1e-4 allowed, as above).  On the bf16 path the
    Ritz vectors come from TF32 operands, 2^-12 each in H relative to its largest entry 1, against the
    smallest leading Ritz value 1/4: 2^-11 / (1/4)."""
    rng = np.random.default_rng(k)
    U4 = np.linalg.qr(rng.standard_normal((m, 4)))[0]
    V4 = np.linalg.qr(rng.standard_normal((n, 4)))[0]
    G = ((U4 * np.linspace(1.0, 0.5, 4)) @ V4.T * scale).astype(np.float32)
    h = _refreshed(m, n, r, k, G, dtype)                 # its stats() raises on a numeric failure
    A = h.selection()[4].double().cpu().numpy()          # bf16: the rounded gradient, rank 4 and small noise
    U = h.basis().double().cpu().numpy()[:, :4]
    h.close()
    U4 = np.linalg.svd(A, full_matrices=False)[0][:, :4]
    assert np.linalg.norm(U4 - U @ (U.T @ U4), 2) <= (2.0 ** -9 if dtype == "bf16" else 1e-4)


@pytest.mark.parametrize("m,n,r,k", [(33, 64, 1, 1), (65, 132, 3, 5), (130, 516, 8, 31), (512, 576, 8, 32), (64, 100, 4, 16)])
def test_scores_use_the_refreshed_basis(m, n, r, k):
    """The step after a refresh reads the copies of Y and Yt that the refresh left (transposed and in fragment
    order): its scores are those of the dense U^T Mbar, as in the allocation-free entry point's own
    test."""
    import torch
    import paper_2507_08784_gb300 as glr
    G = np.random.default_rng(k).standard_normal((m, n)).astype(np.float32)
    h = _refreshed(m, n, r, k, G, "f32", steps=2)
    J, P, Rbar, lam, Mbar = h.selection()
    U = h.basis()
    lam2, J2 = torch.empty_like(lam), torch.empty(r, dtype=torch.int32, device="cuda")
    glr.glr_select_noalloc(U, Mbar, 5, 1, r, lam2, J2)
    torch.cuda.synchronize()
    assert torch.linalg.norm(lam - lam2) <= 1e-4 * torch.linalg.norm(lam2)
    assert sorted(J.tolist()) == sorted(J2.cpu().tolist())
    assert torch.allclose(P, U[:, torch.from_numpy(J.astype(np.int64)).cuda()], rtol=0, atol=1e-5)
    h.close()


@pytest.mark.parametrize("mp,r,k", [(33, 33, 0), (40, 33, 0), (1024, 33, 0), (1024, 512, 0), (1025, 1, 8), (1025, 32, 32),
                                    (1536, 512, 512), (4096, 128, 128), (4096, 512, 512), (16392, 8, 16)])
@pytest.mark.parametrize("kind", ["distinct", "half zero", "all equal"])
def test_step_selection_is_a_stable_top_r(mp, r, k, kind):
    """A step's J is the r largest lambda-bar^2, the lower index first on ties, for the sizes of the radix
    search (m' > 1024 or r > 32; from one score a thread to 17, m' above 16384 among them): under an identity basis a zero row of
    the gradients scores exactly 0, so J has to reach into ties ("half zero") or consists of them.
    Exact: J is compared with a stable sort of the scores that the step used."""
    import torch
    import paper_2507_08784_gb300 as glr
    n = mp + 8
    gen = torch.Generator(device="cuda").manual_seed(mp + r)
    h = glr.GreedyLore(mp, n, r, 1, tau=100, optimizer="msgd", lr=0.01, beta1=0.9, seed=5, basis_rank=k, grad_dtype="f32")
    X = torch.zeros(mp, n, device="cuda")
    h.step([torch.randn(mp, n, device="cuda", generator=gen)], X)        # the refresh; leaves no error behind
    h.set_basis(torch.eye(mp, device="cuda")[:, :k or mp].contiguous())
    G = torch.randn(mp, n, device="cuda", generator=gen)
    if kind == "half zero":
        G[torch.randperm(mp, device="cuda", generator=gen)[:mp - max(1, r // 2)]] = 0.0
    if kind == "all equal":
        G.zero_()
    h.step([G], X)
    J, _, _, lam, _ = h.selection()
    h.close()
    s = (lam * lam).cpu().numpy()
    assert np.count_nonzero(s) == {"distinct": mp, "half zero": max(1, r // 2), "all equal": 0}[kind]
    assert np.array_equal(J, np.sort(np.argsort(-s, kind="stable")[:r]))


@pytest.mark.parametrize("mp,r", [(33, 33), (40, 33), (1024, 33), (1024, 1024), (1025, 1), (1025, 32), (4096, 128),
                                  (4096, 4096), (16384, 300)])
@pytest.mark.parametrize("kind", ["distinct", "half zero", "all equal"])
def test_selection_is_a_stable_top_r(mp, r, kind):
    """J of the allocation-free entry point (its sort of all keys, at any m' and r) = the r largest lambda^2,
    the lower index first on ties: distinct scores, scores tied at 0 that J has to reach into, and all
    tied.  Exact: J is compared with a stable sort of the scores that the kernel returns."""
    import torch
    import paper_2507_08784_gb300 as glr
    gen = torch.Generator(device="cuda").manual_seed(mp + r)
    d = torch.rand(mp, device="cuda", generator=gen) + 0.1
    if kind == "half zero":
        d[torch.randperm(mp, device="cuda", generator=gen)[:mp - max(1, r // 2)]] = 0.0
    if kind == "all equal":
        d.zero_()
    U = torch.zeros(mp, mp, device="cuda")
    U.diagonal().copy_(d)
    Mbar = torch.randn(mp, 8, device="cuda", generator=gen)
    lam, J = torch.empty(mp, device="cuda"), torch.empty(r, dtype=torch.int32, device="cuda")
    glr.glr_select_noalloc(U, Mbar, 9, 3, r, lam, J)
    torch.cuda.synchronize()
    s = (lam * lam).cpu().numpy()
    want = np.sort(np.argsort(-s, kind="stable")[:r])
    assert np.array_equal(np.sort(J.cpu().numpy()), want)
