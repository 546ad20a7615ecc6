"""CUDA path (through the C ABI) against the CPU oracle, element by element, on
seeded inputs that span several tiles with ragged tails.  FP64 path tolerance:
||D_gpu - D_oracle||_F <= 1e-10; integer tile patterns bit-exact."""
import numpy as np
import pytest

from synth import BlockSparse, dense_gapped, from_dense, make_config, to_dense
from tests.helpers import compare, run_gpu, run_oracle

pytestmark = pytest.mark.gpu


def _case(key):
    c = make_config(key)
    return c


@pytest.mark.parametrize("key", [1, "2s", "4s"])
def test_parity_configs(key):
    c = _case(key)
    kw = dict(stop=c["stop"])
    g = run_gpu(c["F"], c["nocc"], c["homo_ub"], c["lumo_lb"], c["tau"], **kw)
    o = run_oracle(c["F"], c["nocc"], c["homo_ub"], c["lumo_lb"], c["tau"], **kw)
    compare(g, o)
    assert g["code"] == 0


def test_parity_cfg1_against_projector():
    c = _case(1)
    g = run_gpu(c["F"], c["nocc"], c["homo_ub"], c["lumo_lb"], 0.0, stop="idempotency")
    import oracle.sp2_oracle as O
    P = O.eig_projector(c["F"], c["nocc"])
    assert np.linalg.norm(g["D"] - P) < 1e-11
    assert abs(np.trace(g["D"]) - c["nocc"]) < 1e-10


@pytest.mark.parametrize("mode", ["sp2", "sp2acc"])
def test_parity_plain_sp2_and_ragged(mode):
    # N = 100: three full tiles and a ragged tail of 4
    d = dense_gapped(100, 37, (-2.0, -0.3), (0.4, 2.0), seed=7)
    g = run_gpu(d["F"], d["nocc"], d["homo_ub"], d["lumo_lb"], 1e-7, mode=mode)
    o = run_oracle(d["F"], d["nocc"], d["homo_ub"], d["lumo_lb"], 1e-7, mode=mode)
    compare(g, o)


@pytest.mark.parametrize("n", [661, 672, 673, 1030])
def test_parity_around_the_split_tile_limit(n):
    # 231 output tiles (also with a ragged tail) take four CTAs a tile, 253 and
    # 561 one; the adjoint's products take the same two kernels
    import paper_1909_12533_gb300 as sp2
    d = dense_gapped(n, n // 2, (-2.0, -0.3), (0.4, 2.0), seed=n)
    kw = dict(stop="idempotency")
    g = run_gpu(d["F"], d["nocc"], d["homo_ub"], d["lumo_lb"], 0.0, record_masks=1, **kw)
    o = run_oracle(d["F"], d["nocc"], d["homo_ub"], d["lumo_lb"], 0.0, **kw)
    compare(g, o)
    if n > 700:
        return
    rng = np.random.default_rng(n)
    W = rng.standard_normal((n, n))
    W = 0.5 * (W + W.T)
    import oracle.sp2_oracle as O
    ctx = sp2.SP2(from_dense(d["F"]), d["nocc"], d["homo_ub"], d["lumo_lb"], 0.0, record_masks=1, **kw)
    ctx.run()
    brow, bcol, val = ctx.backward(from_dense(W, keep_zero_tiles=True))
    ctx.close()
    dF = to_dense(BlockSparse(n=n, brow=brow.cpu().numpy(), bcol=bcol.cpu().numpy(), val=val.cpu().numpy()))
    G = O.adjoint_sp2(d["F"], o, W)
    assert np.linalg.norm(dF - G) <= 1e-10 * np.linalg.norm(G)


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-10), ("split16", 1e-6)])
@pytest.mark.parametrize("nb", [1500, 2502])
def test_many_tile_rows(nb, precision, tol):
    # 1,500 tile rows: the row offsets of a bitmap of 70,500 words come from two
    # launches; 2,502: so do the super-row bitmaps (49,454 words).  F is block
    # diagonal, dense blocks of three tile rows (four kinds, the last one ragged), so
    # D is block diagonal with the projectors of the blocks.
    import paper_1909_12533_gb300 as sp2
    n = 32 * nb - 7
    nblk = nb // 3
    kinds = [dense_gapped(96, 30 + 5 * k, (-2.0, -0.5), (0.5, 2.0), seed=900 + k) for k in range(4)]
    kinds.append(dense_gapped(89, 41, (-2.0, -0.5), (0.5, 2.0), seed=904))
    which = np.arange(nblk) % 4
    which[-1] = 4
    tiles, proj = [], []
    for d in kinds:
        lam, V = np.linalg.eigh(d["F"])
        V = V[:, lam < 0]
        tiles.append(from_dense(d["F"], keep_zero_tiles=True))
        proj.append(from_dense(V @ V.T, keep_zero_tiles=True).val)
    base = 3 * np.arange(nblk, dtype=np.int32)[:, None]
    brow, bcol = (base + t.astype(np.int32) for t in (tiles[0].brow, tiles[0].bcol))
    order = np.lexsort((bcol.ravel(), brow.ravel()))
    F = BlockSparse(n=n, brow=brow.ravel()[order], bcol=bcol.ravel()[order],
                    val=np.concatenate([tiles[k].val for k in which])[order])
    nocc = int(sum(kinds[k]["nocc"] for k in which))
    ctx = sp2.SP2(F, nocc, -0.5, 0.5, 0.0, stop="idempotency", precision=precision)
    st = ctx.run()
    gb, gc, gv = ctx.D_host()
    ctx.close()
    assert st["converged"] and set(st["nnzb_hist"]) == {6 * nblk}
    assert np.array_equal(gb, F.brow) and np.array_equal(gc, F.bcol)
    ref = np.concatenate([proj[k] for k in which])[order]
    assert np.linalg.norm(gv - ref) <= tol, np.linalg.norm(gv - ref)


def test_parity_frobinf_multiple_superblocks():
    c = _case("3s")
    kw = dict(trunc="frobinf", frobinf_part=1024)
    g = run_gpu(c["F"], c["nocc"], c["homo_ub"], c["lumo_lb"], c["tau"], **kw)
    o = run_oracle(c["F"], c["nocc"], c["homo_ub"], c["lumo_lb"], c["tau"], **kw)
    compare(g, o)


def test_parity_gamma_mode():
    c = _case("2s")
    kw = dict(gamma=1e-3)
    g = run_gpu(c["F"], c["nocc"], c["homo_ub"], c["lumo_lb"], 0.0, **kw)
    o = run_oracle(c["F"], c["nocc"], c["homo_ub"], c["lumo_lb"], 0.0, **kw)
    compare(g, o)
    np.testing.assert_allclose(g["stats"]["tau"], o.sched.tau, rtol=1e-14)


@pytest.mark.parametrize("n", [2, 31, 32, 33])
def test_tiny_and_single_tile(n):
    nocc = max(1, n // 2)
    d = dense_gapped(n, nocc, (-1.0, -0.5), (0.5, 1.0), seed=11 + n)
    g = run_gpu(d["F"], d["nocc"], d["homo_ub"], d["lumo_lb"], 0.0, stop="idempotency")
    o = run_oracle(d["F"], d["nocc"], d["homo_ub"], d["lumo_lb"], 0.0, stop="idempotency")
    compare(g, o)
    import oracle.sp2_oracle as O
    assert np.linalg.norm(g["D"] - O.eig_projector(d["F"], d["nocc"])) < 1e-11


def test_block_diagonal_input_keeps_zero_blocks_out():
    # two decoupled molecules-worth blocks: the product pattern stays block diagonal
    a = dense_gapped(64, 32, (-1.0, -0.5), (0.5, 1.0), seed=3)["F"]
    b = dense_gapped(64, 32, (-1.0, -0.5), (0.5, 1.0), seed=4)["F"]
    F = np.zeros((128, 128))
    F[:64, :64] = a
    F[64:, 64:] = b
    Fb = from_dense(F)
    assert Fb.nnzb == 6
    g = run_gpu(Fb, 64, -0.5, 0.5, 0.0, stop="idempotency")
    o = run_oracle(Fb, 64, -0.5, 0.5, 0.0, stop="idempotency")
    compare(g, o)
    assert g["brow"].shape[0] == 6


def test_error_paths():
    import paper_1909_12533_gb300 as sp2
    d = dense_gapped(64, 32, (-1.0, -0.5), (0.5, 1.0), seed=5)
    Fb = from_dense(d["F"])
    # non-finite value
    bad = BlockSparse(n=Fb.n, brow=Fb.brow, bcol=Fb.bcol, val=Fb.val.copy())
    bad.val[1, 3, 4] = np.nan
    with pytest.raises(sp2.SP2Error) as e:
        sp2.SP2(bad, 32, -0.5, 0.5, 0.0)
    assert e.value.code == -4
    # unsorted pattern
    bad = BlockSparse(n=Fb.n, brow=Fb.brow[::-1].copy(), bcol=Fb.bcol[::-1].copy(), val=Fb.val[::-1].copy())
    with pytest.raises(sp2.SP2Error) as e:
        sp2.SP2(bad, 32, -0.5, 0.5, 0.0)
    assert e.value.code == -3
    # lower-triangle tile
    bad = BlockSparse(n=Fb.n, brow=np.array([0, 1, 1], np.int32), bcol=np.array([0, 0, 1], np.int32),
                      val=Fb.val[:3].copy())
    with pytest.raises(sp2.SP2Error) as e:
        sp2.SP2(bad, 32, -0.5, 0.5, 0.0)
    assert e.value.code == -3
    # missing diagonal tile
    bad = BlockSparse(n=Fb.n, brow=np.array([0, 0], np.int32), bcol=np.array([0, 1], np.int32), val=Fb.val[:2].copy())
    with pytest.raises(sp2.SP2Error) as e:
        sp2.SP2(bad, 32, -0.5, 0.5, 0.0)
    assert e.value.code == -3
    # bounds outside the Gershgorin interval
    with pytest.raises(sp2.SP2Error) as e:
        sp2.SP2(Fb, 32, -1e6, 0.5, 0.0)
    assert e.value.code == -2
    # n_max cap reached: NOT_CONVERGED, D still readable
    ctx = sp2.SP2(Fb, 32, d["homo_ub"], d["lumo_lb"], 0.0, n_max_cap=3, stop="idempotency")
    st = ctx.run()
    assert ctx.code == -7 and not st["converged"] and st["n"] == 3
    brow, bcol, val = ctx.D_host()
    assert brow.shape[0] > 0 and np.all(np.isfinite(val))
    ctx.close()


def test_device_input_and_device_view():
    import torch
    import paper_1909_12533_gb300 as sp2
    c = _case("2s")
    Fb = c["F"]

    class T:
        n = Fb.n
        brow = torch.from_numpy(Fb.brow).cuda()
        bcol = torch.from_numpy(Fb.bcol).cuda()
        val = torch.from_numpy(Fb.val).cuda()

    ctx = sp2.SP2(T, c["nocc"], c["homo_ub"], c["lumo_lb"], c["tau"])
    st = ctx.run()
    brow, bcol, val = ctx.D_device()
    hb, hc, hv = ctx.D_host()
    assert np.array_equal(brow.cpu().numpy(), hb) and np.array_equal(bcol.cpu().numpy(), hc)
    assert np.array_equal(val.cpu().numpy(), hv)
    g = run_gpu(Fb, c["nocc"], c["homo_ub"], c["lumo_lb"], c["tau"])
    assert np.array_equal(g["val"], hv)  # host and device inputs give identical results
    assert st["n"] == g["stats"]["n"]
    ctx.close()


def test_run_twice_is_deterministic():
    import paper_1909_12533_gb300 as sp2
    c = _case("4s")
    ctx = sp2.SP2(c["F"], c["nocc"], c["homo_ub"], c["lumo_lb"], c["tau"])
    s1 = ctx.run()
    d1 = ctx.D_host()
    s2 = ctx.run()
    d2 = ctx.D_host()
    ctx.close()
    assert s1["e"] == s2["e"] and s1["t"] == s2["t"]
    assert all(np.array_equal(a, b) for a, b in zip(d1, d2))


def test_contexts_reuse_pooled_memory_and_release():
    # contexts created one after another reuse the library's memory pool; the
    # results do not depend on what the pool held before; release returns it
    import paper_1909_12533_gb300 as sp2
    c = make_config("2s")
    runs = [run_gpu(c["F"], c["nocc"], c["homo_ub"], c["lumo_lb"], c["tau"]) for _ in range(2)]
    assert np.array_equal(runs[0]["val"], runs[1]["val"])
    sp2.sp2_release_memory()
    g = run_gpu(c["F"], c["nocc"], c["homo_ub"], c["lumo_lb"], c["tau"], precision="split16")
    assert g["code"] == 0
    buf = (np.empty(g["brow"].shape[0] + 5, np.int32), np.empty(g["brow"].shape[0] + 5, np.int32),
           np.empty((g["brow"].shape[0] + 5, 32, 32)))
    ctx = sp2.SP2(c["F"], c["nocc"], c["homo_ub"], c["lumo_lb"], c["tau"], precision="split16")
    ctx.run()
    brow, bcol, val = ctx.D_host(buf)
    ctx.close()
    assert np.array_equal(brow, g["brow"]) and np.array_equal(val, g["val"])


# ----------------------------------------------------------------- Step 3 estimates
@pytest.mark.parametrize("key", [1, "2s", "4s"])
def test_homo_lumo_estimates_match_oracle(key):
    # Section 4 Step 3: the estimates come from e_j and t_j, which the GPU path
    # computes to ~1e-10 relative; the same reading of Step 3 then gives the
    # same estimates
    c = _case(key)
    kw = dict(stop=c["stop"])
    g = run_gpu(c["F"], c["nocc"], c["homo_ub"], c["lumo_lb"], c["tau"], **kw)
    o = run_oracle(c["F"], c["nocc"], c["homo_ub"], c["lumo_lb"], c["tau"], **kw)
    _check_estimates(g["stats"], o)


def test_homo_lumo_estimates_near_exact_eigenvalues_plain_sp2():
    # plain SP2 (the paper's first run is unaccelerated, Section 6) on the dense
    # 512 case: the estimates are within 0.02 of the exact homo and lumo
    c = _case(1)
    g = run_gpu(c["F"], c["nocc"], c["homo_ub"], c["lumo_lb"], 0.0, stop="idempotency", mode="sp2")
    st = g["stats"]
    ev = c["eigenvalues"]
    assert st["have_estimates"] == 3
    assert abs(st["homo_est"] - ev[c["nocc"] - 1]) < 0.02
    assert abs(st["lumo_est"] - ev[c["nocc"]]) < 0.02


# ----------------------------------------------------------------- trace-correcting SP2 (Section 1, 6)
def _run_oracle_trace(c, tau, **kw):
    import oracle.sp2_oracle as O
    from tests.helpers import as_blocks
    Fb = as_blocks(c["F"])
    return O.sp2_trace_correcting(to_dense(Fb), c["nocc"], tau=tau, input_pattern=set(zip(Fb.brow.tolist(),
                                                                                           Fb.bcol.tolist())), **kw)


@pytest.mark.parametrize("key", [1, "2s", "4s"])
def test_trace_correcting_matches_oracle(key):
    # no bounds passed (NaN): the polynomial of each iteration comes from trace(X~)
    c = _case(key)
    g = run_gpu(c["F"], c["nocc"], float("nan"), float("nan"), c["tau"], stop=c["stop"], mode="trace")
    o = _run_oracle_trace(c, c["tau"], stop=c["stop"])
    st = g["stats"]
    assert g["code"] == 0 and st["converged"] and o.converged
    assert st["n"] == o.n
    assert st["p"][1:o.n + 1] == o.sched.p[1:o.n + 1]
    assert all(a == 1.0 for a in st["alpha"][1:o.n + 1])
    assert st["tile_triplets"] == o.tile_triplets
    np.testing.assert_allclose(st["e"], o.e, rtol=1e-8, atol=1e-12)
    assert st["nnzb_hist"][: o.n + 1] == [len(k) for k in o.kept[: o.n + 1]]
    assert np.linalg.norm(g["D"] - o.D) <= 1e-10
    _check_estimates(st, o)


def _check_estimates(st, o):
    # Step 3 on the same e_j, t_j gives the same estimates (host arithmetic);
    # end to end the estimates inherit the rounding of e_j, t_j, amplified when
    # the index used sits near convergence (t_j ~ 1e-9 there): 1e-6
    import copy
    import oracle.sp2_oracle as O
    oh, ol = o.estimates
    assert st["have_estimates"] == (1 if oh is not None else 0) | (2 if ol is not None else 0)
    same = copy.copy(o)
    same.e, same.t = list(st["e"]), list(st["t"])
    sh, sl = O.homo_lumo_estimates(same, o.D.shape[0])
    for got, mine, ref in ((st["homo_est"], sh, oh), (st["lumo_est"], sl, ol)):
        if ref is None:
            continue
        assert abs(got - mine) <= 1e-12 * max(1.0, abs(mine))
        assert abs(got - ref) <= 1e-6 * max(1.0, abs(ref))


@pytest.mark.parametrize("key", [1, "2s", "4s"])
def test_two_run_protocol_matches_oracle(key):
    # Section 6: run 1 trace-correcting, run 2 SP2ACC with run 1's estimates
    # widened by 0.1 of the estimated gap; both sides give the same bounds and D
    import oracle.sp2_oracle as O
    import paper_1909_12533_gb300 as sp2
    from tests.helpers import as_blocks
    c = _case(key)
    Fb = as_blocks(c["F"])
    tau1 = 1e-5 if c["tau"] > 0 else 0.0
    (brow, bcol, val), st2, st1, (hub, llb) = sp2.run_two_pass(Fb, c["nocc"], tau1, c["tau"], margin=0.1,
                                                              stop=c["stop"])
    r1, r2, (ohub, ollb) = O.two_run(to_dense(Fb), c["nocc"], tau1, tau=c["tau"], margin=0.1, stop=c["stop"],
                                      input_pattern=set(zip(Fb.brow.tolist(), Fb.bcol.tolist())))
    assert st1["n"] == r1.n and st2["n"] == r2.n
    # the bounds inherit the estimates' sensitivity (see _check_estimates)
    assert abs(hub - ohub) <= 1e-6 and abs(llb - ollb) <= 1e-6
    # run 2 exactly: the oracle's SP2ACC with the bounds the GPU's run 1 produced
    o2 = O.sp2(to_dense(Fb), c["nocc"], hub, llb, tau=c["tau"], stop=c["stop"],
               input_pattern=set(zip(Fb.brow.tolist(), Fb.bcol.tolist())))
    D = to_dense(BlockSparse(n=Fb.n, brow=brow, bcol=bcol, val=val))
    assert st2["n"] == o2.n
    assert np.linalg.norm(D - o2.D) <= 1e-10
    # run 2 against SP2ACC with the recipe's own (Weyl) bounds: iteration counts
    g = run_gpu(Fb, c["nocc"], c["homo_ub"], c["lumo_lb"], c["tau"], stop=c["stop"])
    print(f"config {key}: run 1 (trace) n = {st1['n']}, run 2 (SP2ACC, estimated bounds "
          f"[{hub:.4f}, {llb:.4f}]) n = {st2['n']}, SP2ACC with the recipe's bounds "
          f"[{c['homo_ub']:.4f}, {c['lumo_lb']:.4f}] n = {g['stats']['n']}")


def test_trace_mode_rejects_gamma_and_accepts_nan_bounds():
    import paper_1909_12533_gb300 as sp2
    d = dense_gapped(64, 32, (-1.0, -0.5), (0.5, 1.0), seed=5)
    with pytest.raises(sp2.SP2Error) as e:
        sp2.SP2(from_dense(d["F"]), 32, float("nan"), float("nan"), 0.0, mode="trace", gamma=1e-3)
    assert e.value.code == -1
    with pytest.raises(sp2.SP2Error) as e:
        sp2.SP2(from_dense(d["F"]), 32, float("nan"), float("nan"), 0.0)   # NaN bounds need trace mode
    assert e.value.code == -1


# ----------------------------------------------------------------- general storage (Section 5, 6)
@pytest.mark.parametrize("key,prec", [(1, "fp64"), ("2s", "fp64"), ("4s", "fp64"), ("2s", "split16"),
                                      ("3s", "split16")])
def test_general_storage_matches_symmetric_and_oracle(key, prec):
    # both triangles stored and computed; the selection is made on the upper
    # tiles.  FP64: the upper output tiles are the same products in the same
    # order and the lower ones their exact transposes, so D is the symmetric
    # storage's D bit for bit.  Tensor path: a lower tile is its own set of
    # MMAs whose FP32 group sums (not exact at every size) round in another
    # order, so the iterates agree to rounding only.  The square does the full
    # count of tile products.
    import oracle.sp2_oracle as O
    c = _case(key)
    kw = dict(stop=c["stop"], precision=prec)
    g = run_gpu(c["F"], c["nocc"], c["homo_ub"], c["lumo_lb"], c["tau"], storage="general", **kw)
    s = run_gpu(c["F"], c["nocc"], c["homo_ub"], c["lumo_lb"], c["tau"], **kw)
    assert g["code"] == 0 and g["stats"]["n"] == s["stats"]["n"]
    assert np.array_equal(g["brow"], s["brow"]) and np.array_equal(g["bcol"], s["bcol"])
    if prec == "split16":
        assert np.linalg.norm(g["D"] - s["D"]) <= 1e-8
        o = run_oracle(c["F"], c["nocc"], c["homo_ub"], c["lumo_lb"], c["tau"], stop=c["stop"])
        assert np.linalg.norm(g["D"] - o.D) <= 1e-6
        return
    assert np.array_equal(g["val"], s["val"])
    np.testing.assert_allclose(g["stats"]["e"], s["stats"]["e"], rtol=1e-12, atol=1e-15)
    if prec == "fp64":
        o = run_oracle(c["F"], c["nocc"], c["homo_ub"], c["lumo_lb"], c["tau"], stop=c["stop"])
        assert g["stats"]["n"] == o.n
        nb = g["Fb"].nb
        assert g["stats"]["tile_triplets"] == sum(O.triplets_general(k, nb) for k in o.kept[: o.squares])
        # stored tiles of each X~_j: both triangles of the oracle's upper pattern
        full = [2 * len(k) - sum(1 for i, j in k if i == j) for k in o.kept[: o.n + 1]]
        assert g["stats"]["nnzb_hist"][: o.n + 1] == full
        assert np.linalg.norm(g["D"] - o.D) <= 1e-10


def test_general_storage_rejects_recording_for_the_adjoint():
    import paper_1909_12533_gb300 as sp2
    d = dense_gapped(64, 32, (-1.0, -0.5), (0.5, 1.0), seed=5)
    with pytest.raises(sp2.SP2Error) as e:
        sp2.SP2(from_dense(d["F"]), 32, d["homo_ub"], d["lumo_lb"], 0.0, storage="general", record_masks=1)
    assert e.value.code == -1


# ----------------------------------------------------------------- mixed-norm truncation in the expansion
@pytest.mark.parametrize("key,part", [("2s", 512), ("4s", 1024), ("3s", 1024)])
def test_parity_mixed_norm_truncation(key, part):
    c = _case(key)
    kw = dict(trunc="mixed", frobinf_part=part)
    g = run_gpu(c["F"], c["nocc"], c["homo_ub"], c["lumo_lb"], c["tau"], **kw)
    o = run_oracle(c["F"], c["nocc"], c["homo_ub"], c["lumo_lb"], c["tau"], **kw)
    compare(g, o)
    f = run_oracle(c["F"], c["nocc"], c["homo_ub"], c["lumo_lb"], c["tau"], trunc="frobinf", frobinf_part=part)
    print(f"config {key}: stored tiles of D, mixed norm {len(o.kept[o.n])}, Frob-Inf {len(f.kept[f.n])}")
