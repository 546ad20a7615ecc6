"""Truncation step (Eq. (8)) through sp2_truncate against the oracle's selection:
bit-exact keep flags, including exact ties, tau = 0 and the two extremes."""
import numpy as np
import pytest

import oracle.sp2_oracle as O
from synth import BlockSparse, from_dense, to_dense

pytestmark = pytest.mark.gpu


def _decaying(n, seed, ties=False):
    rng = np.random.default_rng(seed)
    A = rng.standard_normal((n, n))
    A = 0.5 * (A + A.T)
    d = np.abs(np.subtract.outer(np.arange(n), np.arange(n)))
    A *= np.exp(-d / 40.0)
    X = from_dense(A, keep_zero_tiles=True)
    if ties:
        # several tiles with bit-identical values (equal norms): the index decides
        off = np.nonzero(X.brow != X.bcol)[0]
        src = X.val[off[3]].copy()
        for k in off[5:40:3]:
            X.val[k] = src * 1e-3
        # rows and columns past n are padding and stay zero
        r0 = n - 32 * (X.nb - 1)
        X.val[X.bcol == X.nb - 1, :, r0:] = 0.0
        X.val[X.brow == X.nb - 1, r0:, :] = 0.0
    return X


def _oracle_keep(X, tau, mode, part):
    Xd = to_dense(X)
    pattern = set(zip(X.brow.tolist(), X.bcol.tolist()))
    _, kept, _ = O.truncate_select(Xd, tau, mode, part=part, pattern=pattern)
    ks = set(kept)
    return np.array([1 if (i, j) in ks else 0 for i, j in zip(X.brow.tolist(), X.bcol.tolist())], np.int32)


@pytest.mark.parametrize("mode,part", [("frobenius", 4096), ("frobinf", 64), ("frobinf", 128)])
@pytest.mark.parametrize("tau", [0.0, 1e-6, 1e-3, 0.1])
@pytest.mark.parametrize("ties", [False, True])
def test_keep_flags_bit_exact(mode, part, tau, ties):
    import paper_1909_12533_gb300 as sp2
    X = _decaying(331, 17, ties)      # 11 tile rows, ragged tail of 11
    g = sp2.sp2_truncate(X, tau, mode, part)
    o = _oracle_keep(X, tau, mode, part)
    assert np.array_equal(g, o), np.nonzero(g != o)


def test_zero_tiles_and_extremes():
    import paper_1909_12533_gb300 as sp2
    X = _decaying(200, 3)
    X.val[2] = 0.0
    X.val[7] = 0.0
    keep = sp2.sp2_truncate(X, 0.0, "frobenius")
    assert keep.sum() == X.nnzb - 2 and keep[2] == 0 and keep[7] == 0
    assert sp2.sp2_truncate(X, 1e6, "frobenius").sum() == 0          # everything fits
    assert sp2.sp2_truncate(X, 1e-300, "frobenius").sum() == X.nnzb - 2


def test_device_input_matches_host_input():
    import torch
    import paper_1909_12533_gb300 as sp2
    X = _decaying(480, 9)

    class T:
        n = X.n
        brow = torch.from_numpy(X.brow).cuda()
        bcol = torch.from_numpy(X.bcol).cuda()
        val = torch.from_numpy(X.val).cuda()

    kd = sp2.sp2_truncate(T, 1e-4, "frobinf", 128).cpu().numpy()
    kh = sp2.sp2_truncate(X, 1e-4, "frobinf", 128)
    assert np.array_equal(kd, kh)


@pytest.mark.parametrize("n", [2016, 2048, 2017])
@pytest.mark.parametrize("mode", ["frobenius", "frobinf"])
@pytest.mark.parametrize("tau", [0.0, 1e-4, 0.3])
def test_keep_flags_around_one_cta_limit(n, mode, tau):
    """2016 upper tiles (nb = 63) take the one-CTA select, 2080 (nb = 64, also
    with a ragged tail) the cluster's passes; both match the oracle bit for bit."""
    import paper_1909_12533_gb300 as sp2
    X = _decaying(n, 5, ties=True)
    X.val[11] = 0.0
    g = sp2.sp2_truncate(X, tau, mode, 4096)
    o = _oracle_keep(X, tau, mode, 4096)
    assert np.array_equal(g, o), np.nonzero(g != o)


@pytest.mark.parametrize("n,part", [(331, 32), (5900, 3008)])
@pytest.mark.parametrize("tau", [0.0, 1e-3, 1e3])
def test_keep_flags_of_both_segment_selects(n, part, tau):
    """Frob-Inf with 66 one-tile segments (one CTA each) and with three segments
    of 5,735 tiles on average (a cluster each), equal norms among them."""
    import paper_1909_12533_gb300 as sp2
    X = _decaying(n, 23, ties=True)
    X.val[11] = 0.0
    g = sp2.sp2_truncate(X, tau, "frobinf", part)
    o = _oracle_keep(X, tau, "frobinf", part)
    assert np.array_equal(g, o), np.nonzero(g != o)


@pytest.mark.parametrize("n,mode,part", [(2030, "frobenius", 4096), (500, "frobenius", 4096), (2030, "frobinf", 256),
                                         (5900, "frobinf", 3008)])
@pytest.mark.parametrize("tau", [0.0, 1e-3, 1e3])
def test_tiles_with_nan_are_kept(n, mode, part, tau):
    """A tile whose norm is a NaN fits into no budget and ranks above every finite
    one: the flags are those of the same tiles with a huge norm instead.  Several
    NaNs per selection, in the one-CTA select, both segment selects and the cluster."""
    import paper_1909_12533_gb300 as sp2
    X = _decaying(n, 31)
    bad = np.linspace(1, X.nnzb - 2, 9).astype(int)
    Y = BlockSparse(n=n, brow=X.brow, bcol=X.bcol, val=X.val.copy())
    X.val[bad, 3, 5] = np.nan
    Y.val[bad, 3, 5] = 1e100
    g = sp2.sp2_truncate(X, tau, mode, part)
    o = _oracle_keep(Y, tau, mode, part)
    assert np.array_equal(g, o), np.nonzero(g != o)
    assert g[bad].all()


@pytest.mark.parametrize("n", [500, 2100])
def test_tau_with_a_subnormal_square_drops_zero_tiles_only(n):
    import paper_1909_12533_gb300 as sp2
    X = _decaying(n, 7)
    X.val[3:9] = 0.0
    g = sp2.sp2_truncate(X, 1e-155, "frobenius")
    assert not g[3:9].any() and g.sum() == X.nnzb - 6


def test_more_super_blocks_than_a_32_bit_segment_index_holds():
    """46,400 super-rows of 32 rows (46,400^2 > 2^31 segments), a block-tridiagonal
    set with one element a tile: every segment is one tile of weight 1."""
    import torch
    import paper_1909_12533_gb300 as sp2
    nb = 46400
    brow = np.repeat(np.arange(nb, dtype=np.int32), 2)[:-1]
    bcol = brow.copy()
    bcol[1::2] += 1
    a = np.random.default_rng(46).uniform(0.5, 1.5, brow.size)

    class T:
        n = 32 * nb - 5

    T.brow = torch.from_numpy(brow).cuda()
    T.bcol = torch.from_numpy(bcol).cuda()
    T.val = torch.zeros(brow.size, 32, 32, dtype=torch.float64, device="cuda")
    T.val[:, 0, 0] = torch.from_numpy(a).cuda()
    tau = 3.0
    g = sp2.sp2_truncate(T, tau, "frobinf", 32).cpu().numpy()
    m = np.full(nb, 3)
    m[[0, -1]] = 2
    beta = tau / np.maximum(m[brow], m[bcol])
    keep = np.ceil((a * a) * (2.0 ** 36 / (beta * beta))) > 2.0 ** 36
    assert np.array_equal(g, keep.astype(np.int32)) and 0 < g.sum() < g.size
    sp2.load().sp2_release_memory()      # 26 GB of segment tables


@pytest.mark.parametrize("n,mode,part", [(2030, "frobinf", 256), (331, "frobinf", 32), (5900, "frobinf", 3008),
                                         (2030, "frobenius", 4096)])
def test_tiles_in_any_order_and_below_the_diagonal(n, mode, part):
    """The selection does not depend on the order of the tiles, nor on which of the
    two places (I, J), (J, I) an off-diagonal tile is given at (its norm and its
    segment's budget are the same): shuffled tiles, tiles stored below the
    diagonal, and both, in the one-CTA, the cluster and the small select."""
    import paper_1909_12533_gb300 as sp2
    X = _decaying(n, 29)
    o = _oracle_keep(X, 1e-2, mode, part)
    pt = part // 32 if mode == "frobinf" else 1
    below = (X.brow // pt + X.bcol // pt) % 3 == 0      # whole segments: each has its own budget
    perm = np.random.default_rng(3).permutation(X.nnzb)
    for order, swap in ((perm, False), (np.arange(X.nnzb), True), (perm, True)):
        s = below & swap
        Y = BlockSparse(n=n, brow=np.where(s, X.bcol, X.brow)[order], bcol=np.where(s, X.brow, X.bcol)[order],
                        val=X.val[order])
        g = sp2.sp2_truncate(Y, 1e-2, mode, part)
        assert np.array_equal(g, o[order]), (order is perm, swap, np.nonzero(g != o[order]))


@pytest.mark.parametrize("part,tau", [(64, 0.3), (256, 0.3), (352, 0.3), (384, 0.3), (384, 1e-3)])
def test_keep_flags_of_segments_around_the_direct_limit(part, tau):
    """Segments of at most 4, 64, 121 and 144 tiles (the diagonal ones 3, 36, 66 and
    78): up to 64 tiles are compared with one another, more take histograms; equal
    norms and zero tiles among them."""
    import paper_1909_12533_gb300 as sp2
    X = _decaying(2030, 37, ties=True)
    X.val[[11, 400, 401, 900]] = 0.0
    g = sp2.sp2_truncate(X, tau, "frobinf", part)
    o = _oracle_keep(X, tau, "frobinf", part)
    assert np.array_equal(g, o), np.nonzero(g != o)
    assert 0 < g.sum() < X.nnzb


@pytest.mark.parametrize("mode,part", [("frobenius", 4096), ("frobinf", 704), ("frobinf", 1056)])
@pytest.mark.parametrize("classes", [1, 2, 6])
def test_many_tiles_of_equal_norm(mode, part, classes):
    """All norms are equal, or one of a few that alternate along the rows (what a
    periodic system has): the lanes of a warp share their bins, and the cut lies
    among equal norms, so the index decides."""
    import paper_1909_12533_gb300 as sp2
    n = 2100
    nb = (n + 31) // 32
    i, j = np.triu_indices(nb)
    val = np.zeros((i.size, 32, 32))
    val[:, 0, 0] = 1.0 + 0.25 * ((j - i) % classes)
    X = BlockSparse(n=n, brow=i.astype(np.int32), bcol=j.astype(np.int32), val=val)
    for tau in (3.0, 31.0, 61.0):
        g = sp2.sp2_truncate(X, tau, mode, part)
        o = _oracle_keep(X, tau, mode, part)
        assert np.array_equal(g, o), (tau, np.nonzero(g != o))
        assert 0 < g.sum() < g.size


# ----------------------------------------------------------------- mixed norm (Section 3)
@pytest.mark.parametrize("part", [64, 128, 4096])
@pytest.mark.parametrize("tau", [0.0, 1e-6, 1e-3, 0.1])
@pytest.mark.parametrize("ties", [False, True])
def test_mixed_keep_flags_bit_exact(part, tau, ties):
    # the same integer block sums, bisection and power-step bound on both sides
    import paper_1909_12533_gb300 as sp2
    X = _decaying(331, 17, ties)
    g = sp2.sp2_truncate(X, tau, "mixed", part)
    o = _oracle_keep(X, tau, "mixed", part)
    assert np.array_equal(g, o), np.nonzero(g != o)


@pytest.mark.parametrize("n,part", [(2017, 256), (4000, 128)])
def test_mixed_keep_flags_larger_and_norm_bound(n, part):
    # dropped error: ||E||_2 <= ||E||_m <= tau (exact mixed norm by eigvalsh)
    import paper_1909_12533_gb300 as sp2
    X = _decaying(n, 6)
    tau = 1e-3
    g = sp2.sp2_truncate(X, tau, "mixed", part)
    o = _oracle_keep(X, tau, "mixed", part)
    assert np.array_equal(g, o), np.nonzero(g != o)
    Xd = to_dense(X)
    dropped = [(i, j) for i, j, k in zip(X.brow.tolist(), X.bcol.tolist(), g.tolist()) if not k]
    E = Xd - O.apply_drop(Xd, dropped)
    e = np.append(np.arange(0, n, part), n)
    k = len(e) - 1
    Bm = np.array([[np.linalg.norm(E[e[a]:e[a + 1], e[b]:e[b + 1]]) for b in range(k)] for a in range(k)])
    m = float(np.abs(np.linalg.eigvalsh(Bm)).max())
    assert 0 < len(dropped) and m <= tau * (1 + 1e-12)
