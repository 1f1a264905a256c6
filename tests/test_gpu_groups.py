"""Grouped steps against single steps, bit for bit, at the sizes where the grouping itself can go
wrong (marked gpu): more matrices than one launch takes, basis widths on both sides of a buffer
pitch, sizes that fit no tile, both orientations."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()


def _group_equals_single(mats, steps=3, N=2, dtype="f32", **kw):
    """mats: (m, n, r, basis_rank) each."""
    import torch
    import paper_2507_08784_gb300 as glr
    mk = lambda: [glr.GreedyLore(m, n, r, N, seed=70 + j, basis_rank=k, grad_dtype=dtype, **kw)
                  for j, (m, n, r, k) in enumerate(mats)]
    solo, grp = mk(), mk()
    Xs = [torch.zeros(m, n, device="cuda") for m, n, _, _ in mats]
    Xg = [torch.zeros(m, n, device="cuda") for m, n, _, _ in mats]
    tdt = torch.float32 if dtype == "f32" else torch.bfloat16
    gen = torch.Generator(device="cuda").manual_seed(11)
    for t in range(steps):
        G = [[torch.randn(m, n, device="cuda", generator=gen).to(tdt) for _ in range(N)] for m, n, _, _ in mats]
        for h, g, x in zip(solo, G, Xs):
            h.step(g, x)
        glr.glr_step_group(grp, G, Xg)
        torch.cuda.synchronize()
        for j in range(len(mats)):
            assert torch.equal(Xs[j], Xg[j]), (t, j, mats[j])
            assert np.array_equal(solo[j].selection()[0], grp[j].selection()[0])
            assert torch.equal(solo[j].error(0), grp[j].error(0))
    for h in solo + grp:
        h.close()


def test_refreshes_of_mixed_widths_and_more_than_a_launch():
    """Refreshes with k <= 16 and k <= 32 keep partials of different pitches, and a launch takes 32
    matrices: 36 matrices with k = 8, 16, 20 and 32 refresh in one call."""
    ks = (8, 16, 20, 32)
    mats = [(40 + 8 * (j % 5), 96 + 4 * (j % 7), 4, ks[j % 4]) for j in range(36)]
    _group_equals_single(mats, tau=2, optimizer="msgd", lr=0.05, beta1=0.9)


@pytest.mark.parametrize("opt", ["msgd", "adam"])
def test_ragged_sizes_grouped(opt):
    """The unfused steps of several matrices share their launches: sizes on both sides of the 64 x 64 tiles
    and of the products' K slices, rows of odd length, both orientations, the full basis beside
    truncated ones."""
    mats = [(20, 31, 3, 8), (63, 65, 5, 12), (64, 129, 4, 16), (129, 63, 7, 24), (333, 777, 9, 24),
            (777, 333, 6, 33), (65, 257, 5, 0), (129, 65, 3, 0)]
    _group_equals_single(mats, tau=2, optimizer=opt, lr=0.01, beta1=0.9)


def test_tcgen05_sizes_grouped():
    """m' = 136 and 200 end in a 128-row tile whose lower half holds no row, k = 20 to 132 take the
    small and the blocked eigenproblem beside each other."""
    mats = [(136, 264, 16, 20), (264, 136, 16, 64), (200, 328, 32, 68), (192, 136, 20, 128), (256, 520, 16, 132)]
    _group_equals_single(mats, dtype="bf16", tau=2, optimizer="adam", lr=0.01, beta1=0.9, beta2=0.99)


@pytest.mark.parametrize("m,n,r,k,dtype,opt", [(64, 576, 8, 16, "f32", "msgd"), (65, 131, 4, 12, "f32", "adam"),
                                               (64, 128, 4, 0, "f32", "msgd"), (256, 704, 32, 64, "bf16", "adam")])
@pytest.mark.parametrize("t", [2, 3])
def test_step_recorded_into_a_graph(m, n, r, k, dtype, opt, t):
    """A step (t = 2: a refresh, 3: compressed) recorded on a capturing stream with new gradient buffers,
    replayed, and followed by an ordinary step: the same bits as ordinary steps throughout.  The
    tile-copy descriptors of the recorded step's gradients have to outlive the call that recorded
    them."""
    import torch
    import paper_2507_08784_gb300 as glr
    N = 4
    tdt = torch.float32 if dtype == "f32" else torch.bfloat16
    gen = torch.Generator(device="cuda").manual_seed(3)
    kw = dict(tau=2, optimizer=opt, lr=0.01, beta1=0.9, beta2=0.99, basis_rank=k, seed=4, grad_dtype=dtype)
    a, b = glr.GreedyLore(m, n, r, N, **kw), glr.GreedyLore(m, n, r, N, **kw)
    Xa, Xb = torch.zeros(m, n, device="cuda"), torch.zeros(m, n, device="cuda")
    G = [[torch.randn(m, n, device="cuda", generator=gen).to(tdt) for _ in range(N)] for _ in range(t + 2)]
    for g in G:
        a.step(g, Xa)
    for g in G[:t]:
        b.step(g, Xb)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        b.step(G[t], Xb)
    graph.replay()
    torch.cuda.synchronize()
    b.step(G[t + 1], Xb)
    torch.cuda.synchronize()
    assert torch.equal(Xa, Xb)
    a.close()
    b.close()


def _kernel_nodes(run):
    """Kernels that run() launches on a capturing stream, counted from the graph it leaves."""
    import ctypes
    import torch
    cu = ctypes.CDLL("libcuda.so.1")
    stream = torch.cuda.Stream()
    st, graph, n, kind = ctypes.c_void_p(stream.cuda_stream), ctypes.c_void_p(), ctypes.c_size_t(0), ctypes.c_int(0)

    def check(rc):
        assert rc == 0, rc

    with torch.cuda.stream(stream):
        check(cu.cuStreamBeginCapture_v2(st, 2))               # relaxed
        try:
            run()
        finally:
            rc = cu.cuStreamEndCapture(st, ctypes.byref(graph))
        check(rc)
    check(cu.cuGraphGetNodes(graph, None, ctypes.byref(n)))
    nodes = (ctypes.c_void_p * n.value)()
    check(cu.cuGraphGetNodes(graph, nodes, ctypes.byref(n)))
    kernels = 0
    for node in nodes:
        check(cu.cuGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)))
        kernels += kind.value == 0                             # CU_GRAPH_NODE_TYPE_KERNEL
    check(cu.cuGraphDestroy(graph))
    return kernels


@pytest.mark.parametrize("dtype,opt,mats", [
    # grouped k <= 32 refreshes beside the larger factors and the eigenproblems' size classes
    ("f32", "msgd", [(40, 96, 4, 8), (64, 576, 8, 32), (100, 132, 4, 40), (200, 240, 4, 130), (280, 300, 4, 264)]),
    # no multiple of 4: the unfused step and the ungrouped refresh with K slices; full bases up to and above 256
    ("f32", "adam", [(65, 131, 4, 12), (63, 777, 5, 20), (129, 65, 3, 0), (300, 310, 4, 0)]),
    ("f32", "adamw", [(65, 131, 4, 12)]),
    ("f32", "amsgrad", [(64, 128, 4, 0)]),
    # tcgen05: whole and sliced products, each class of eigenproblem, Gram matrices of several row chunks
    ("bf16", "adam", [(136, 264, 16, 20), (200, 328, 16, 68), (256, 4104, 16, 64), (520, 1032, 16, 64), (264, 520, 16, 256)]),
])
def test_launch_counts_are_the_kernels_launched(dtype, opt, mats):
    """glr_stats.launches against the kernel nodes of the recorded step, for a refresh and a compressed step
    (sizes whose products stay below the library's threshold)."""
    import torch
    import paper_2507_08784_gb300 as glr
    tdt = torch.float32 if dtype == "f32" else torch.bfloat16
    hs = [glr.GreedyLore(m, n, r, 2, seed=j, basis_rank=k, grad_dtype=dtype, tau=2, optimizer=opt, lr=0.01, beta1=0.9,
                         beta2=0.99) for j, (m, n, r, k) in enumerate(mats)]
    X = [torch.zeros(m, n, device="cuda") for m, n, _, _ in mats]
    G = [[torch.randn(m, n, device="cuda").to(tdt) for _ in range(2)] for m, n, _, _ in mats]
    for _ in range(2):
        glr.glr_step_group(hs, G, X)
    torch.cuda.synchronize()
    for what in ("refresh", "compressed"):
        before = sum(h.stats()["launches"] for h in hs)
        kernels = _kernel_nodes(lambda: glr.glr_step_group(hs, G, X))
        assert sum(h.stats()["launches"] for h in hs) - before == kernels, what
    for h in hs:
        h.close()


def test_recording_again_keeps_no_more():
    """A handle keeps the tile-copy descriptors that recorded steps read (N + 1 of 128 bytes a recording);
    recordings of the same buffers share them: the process's allocated bytes grow by less than a
    recording's descriptors."""
    import ctypes
    import torch
    import paper_2507_08784_gb300 as glr

    class Mallinfo2(ctypes.Structure):
        _fields_ = [(f, ctypes.c_size_t) for f in ("arena", "ordblks", "smblks", "hblks", "hblkhd", "usmblks", "fsmblks",
                                                   "uordblks", "fordblks", "keepcost")]
    libc = ctypes.CDLL(None)
    libc.mallinfo2.restype = Mallinfo2
    N = 8
    h = glr.GreedyLore(256, 704, 32, N, seed=1, basis_rank=64, grad_dtype="bf16", tau=1 << 20, optimizer="adam", lr=0.01)
    X = torch.zeros(256, 704, device="cuda")
    G = [torch.randn(256, 704, device="cuda").to(torch.bfloat16) for _ in range(N)]
    for _ in range(2):
        h.step(G, X)
    torch.cuda.synchronize()
    used = []
    for _ in range(4):
        for _ in range(250):
            _kernel_nodes(lambda: h.step(G, X))
        used.append(libc.mallinfo2().uordblks)
    h.close()
    assert min(b - a for a, b in zip(used, used[1:])) < 250 * (N + 1) * 128 / 2
