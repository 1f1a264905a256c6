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
