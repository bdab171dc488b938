"""The dense linear algebra behind Eq. 3-5 / 3-6 (Sec. 3.3.1) at the sizes where a tile, a register
layout or a cluster ends, against the float64 oracle, through the C ABI."""
import numpy as np
import pytest
import torch

from oracle import ipgs_oracle as orc
from paper_2503_10501_b200 import binding as tcb
from paper_2503_10501_b200 import inputs
import parity_util as pu

pytestmark = pytest.mark.gpu


def _inputs(N, d, rank, seed, noise, batch=2):
    """O of numerical rank `rank` (singular values geometric 1 .. 0.03), and attention."""
    rng = np.random.default_rng(seed)
    u = np.linalg.qr(rng.standard_normal((batch, N, rank)))[0]
    w = np.linalg.qr(rng.standard_normal((batch, d, rank)))[0]
    s = np.geomspace(100.0, 3.0, rank)
    O = (u * s) @ w.transpose(0, 2, 1) + noise * rng.standard_normal((batch, N, d))
    A = rng.random((batch, 1, 3, N))
    return O.astype(np.float32), A.astype(np.float32)


def _check(N, d, rank, rank_cap, seed, noise=1e-6):
    O, A = _inputs(N, d, rank, seed, noise)
    p = tcb.Params(batch=2, n_tokens=N, d_model=d, n_heads=1, head_dim=8, n_query=3, keep=1,
                   rank_tol=2e-3, dtype="f32", rank_cap=rank_cap)
    g = tcb.tc_score(p, torch.from_numpy(O).cuda(), torch.from_numpy(A).cuda())
    torch.cuda.synchronize()
    # (the sweeps of the full solve may go on over rounding noise until they are stopped)
    assert not g["img_status"].any() or (rank_cap == 0 and set(g["img_status"].tolist()) <= {0, 4})
    for b in range(2):
        pu.check_scores({k: v[b].cpu().numpy() for k, v in g.items()}, orc.score(O[b], A[b], 0.5, 2e-3), 2e-3)


# orders of the tridiagonal solver: the smallest, register layouts and cluster sizes from both sides,
# and one that no layout fills
@pytest.mark.parametrize("N", [3, 4, 7, 32, 33, 64, 65, 96, 97, 128, 129, 144, 145, 160, 161, 192, 193, 256,
                               257, 320, 321, 384, 385, 448, 449, 500, 512, 513, 576, 577, 640, 641, 768])
def test_eigenvalues_of_every_layout(N):
    O, _ = _inputs(N, 832, max(2, min(N // 3, 200)), N, 1e-6)
    p = tcb.Params(batch=2, n_tokens=N, d_model=832, n_heads=1, head_dim=8, n_query=3, keep=1, rank_tol=2e-3, dtype="f32")
    g = tcb.tc_rank(p, torch.from_numpy(O).cuda())
    torch.cuda.synchronize()
    assert not g["img_status"].any()
    for b in range(2):
        s = np.linalg.svd(O[b].astype(np.float64), compute_uv=False)
        assert np.allclose(g["sigma"][b].cpu().numpy(), s, rtol=1e-4, atol=1e-3 * s[0])
        assert int(g["rank"][b]) == int((s > 2e-3 * s[0]).sum())


# full solves: one block, W in the shared memory of clusters of either size (every column length, byes), out of L2
@pytest.mark.parametrize("N", [3, 4, 33, 96, 97, 128, 129, 193, 257, 320, 321, 449, 576, 577, 672, 673, 700])
def test_full_solve(N):
    _check(N, 832, max(2, min(N // 3, 200)), 0, seed=N)


# subspaces: widths that no product tile fills, around one and several Cholesky blocks and the width the
# float32 chain takes over at; token counts that are no multiple of four; a bound that leaves no
# subspace once it is rounded up
@pytest.mark.parametrize("N,rank_cap", [(97, 30), (131, 47), (203, 64), (330, 100), (333, 177), (401, 193), (450, 209), (460, 224), (520, 304),
                                        (601, 385), (801, 577), (900, 640), (902, 641), (120, 111), (2881, 150)])
def test_subspace_of_every_width(N, rank_cap):
    _check(N, 1000, max(8, min(rank_cap - 16, rank_cap * 3 // 4, 200)), rank_cap, seed=N, noise=1e-3)


@pytest.mark.parametrize("B,N,d", [(1, 3, 64), (1, 64, 32), (2, 100, 36), (1, 128, 384), (3, 132, 388), (1, 133, 100), (1, 576, 1024), (9, 260, 416)])
def test_float32_gram(B, N, d):
    g = torch.Generator().manual_seed(N * d)
    O = torch.randn(B, N, d, generator=g)
    O[:, N // 2] = O[:, 0]   # identical rows have identical products
    p = tcb.Params(batch=B, n_tokens=N, d_model=d, n_heads=1, head_dim=d, n_query=1, keep=1, rank_tol=0.0, dtype="f32")
    G = tcb.tc_gram(p, O.cuda()).cpu()
    norm = O.double().norm(dim=2)
    err = (G.double() - O.double() @ O.double().mT).abs() / (norm[:, :, None] * norm[:, None, :])
    assert err.max() < 2e-6
    assert torch.equal(G, G.mT)
    assert torch.equal(G[:, N // 2], G[:, 0])


@pytest.mark.parametrize("keep", [40, 97, 98])   # survivors just under, at and above three quarters of the tokens
@pytest.mark.parametrize("where", ["pinned", "pageable", "middle of a pinned block"])
def test_host_rows_gathered_or_copied(keep, where):
    cfg = inputs.tiny_config(n_tokens=195, d_model=64, n_heads=3, head_dim=16, n_query=5, keep=keep, rank=30, dtype="f16",
                             batch=3, seed=5, noise=0.3, rank_tol=0.0)
    p = tcb.Params(batch=3, n_tokens=195, d_model=64, n_heads=3, head_dim=16, n_query=5, keep=keep, rank_tol=0.0, dtype="f16")
    data = inputs.make_batch(cfg)
    t = [torch.from_numpy(np.ascontiguousarray(data[k])) for k in "OAXKV"]
    ref = [None if x is None else x.cpu() for x in tcb.tc_carve(p, *(x.cuda() for x in t), ws=tcb.workspace(p))]
    if where == "pinned":
        t = [x.pin_memory() for x in t]
    elif where != "pageable":
        def inside(x):
            y = torch.empty(x.numel() + 64, dtype=x.dtype, pin_memory=True)[32:32 + x.numel()].view(x.shape)
            return y.copy_(x)
        t = [inside(x) for x in t]
    out = tuple(torch.empty(r.shape, dtype=r.dtype, pin_memory=True) for r in ref)
    ws = tcb.workspace(p, host=True)
    tcb.tc_carve_host(p, *t, out, ws)
    torch.cuda.synchronize()
    for a, b in zip(ref, out):
        assert torch.equal(a, b)
