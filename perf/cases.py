"""The calls whose speed counts, with their inputs, work and tolerances.

Every case is one whole use of the public Python entry points: a Fock matrix F
goes in, the density matrix D (or the gradient dL/dF, or the truncation's keep
flags) comes out.  The inputs follow the recipes of ``synth/fock.py`` (the same
distributions and sizes, drawn with torch on the device): dense matrices with a
prescribed spectrum, water-like clusters of 24 basis functions a molecule, and
helix-like chains of 64 basis functions a residue.

A case is a dict with ``kind`` and the parameters of that kind:

* ``dense``     n, gap (half of it on either side of 0), prec, slices, stop
* ``water``     nmol, tau, prec, trunc, part, out ("tiles": D's tiles into
                device buffers of the caller, "dense": D as a dense device
                matrix, "host": F from host arrays and D's tiles into
                page-locked host buffers)
* ``twopass``   nmol, tau, tau1 (F a dense device matrix, no eigenvalue bounds
                known: two runs, D dense)
* ``helix``     nres, tau, prec, autograd (gradient of trace(D W) through
                ``SP2Function`` instead of ``SP2.backward``)
* ``truncate``  nb, tau, trunc, part (one truncation of the full upper tile set
                of nb tile rows)

D's number of tiles follows from the values, so the callers' buffers are larger
than D and are returned whole with the number of tiles in use.
"""
from __future__ import annotations

import ctypes
import math

import torch

import paper_1909_12533_gb300 as sp2

B = 32          # tile edge
WATER = 24      # basis functions of a molecule
HELIX = 64      # basis functions of a residue
DENSITY = 0.0334


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # the smallest whole run: a dense matrix of a small molecule, everything in
        # FP64 (the default precision); launches and round trips count
        dict(name="dense512", kind="dense", n=512, gap=1.0, prec="fp64", slices=0, stop="idempotency"),
        # a small dense matrix with a narrow gap and a ragged last tile, on the
        # tensor cores with the final squares in FP64
        dict(name="dense1000-tail", kind="dense", n=1000, gap=0.05, prec="split16", slices=5, stop="idempotency"),
        # the tile-GEMM case: dense, narrow gap, five slices, every square on the
        # tensor cores
        dict(name="dense4096-k5", kind="dense", n=4096, gap=0.05, prec="split16", slices=5, stop="parameterless"),
        # a small cluster in FP64, D wanted as a dense matrix (ragged last tile)
        dict(name="water101-fp64", kind="water", nmol=101, tau=1e-6, prec="fp64", trunc="frobenius", part=4096,
             out="dense"),
        # a small cluster from a host program: F from host arrays, D back to the host
        dict(name="water101-host", kind="water", nmol=101, tau=1e-6, prec="split16", trunc="frobenius", part=4096,
             out="host"),
        # an ordinary cluster, N = 24,000, F and D on the device
        dict(name="water1000", kind="water", nmol=1000, tau=1e-6, prec="split16", trunc="frobenius", part=4096,
             out="tiles"),
        # a large cluster at the looser threshold, N = 96,000
        dict(name="water4000", kind="water", nmol=4000, tau=1e-5, prec="split16", trunc="frobenius", part=4096,
             out="tiles"),
        # the truncation norm that adds up over super-rows, N = 19,200
        dict(name="water800-frobinf", kind="water", nmol=800, tau=1e-5, prec="split16", trunc="frobinf", part=4096,
             out="tiles"),
        # no eigenvalue bounds known: a trace-correcting run, then the accelerated one
        dict(name="water400-twopass", kind="twopass", nmol=400, tau=1e-6, tau1=1e-5),
        # a long chain with its gradient, N = 64,000: forward, then the reverse sweep
        dict(name="helix1000-grad", kind="helix", nres=1000, tau=1e-6, prec="split16", autograd=False),
        # a short chain with its gradient in FP64, through the autograd function
        dict(name="helix32-autograd", kind="helix", nres=32, tau=1e-6, prec="fp64", autograd=True),
        # one truncation of a large tile set by itself
        dict(name="truncate-180k", kind="truncate", nb=600, tau=1e-2, trunc="frobenius", part=4096),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["dense", "dense", "water", "water", "water", "twopass", "helix", "truncate"])
    if kind == "dense":
        if rng.random() < 0.4:
            return dict(kind=kind, n=_log(rng, 96, 1024), gap=rng.choice([1.0, 0.3]), prec="fp64", slices=0,
                        stop="idempotency")
        if rng.random() < 0.5:
            return dict(kind=kind, n=_log(rng, 96, 1024), gap=rng.choice([0.3, 0.05]), prec="split16", slices=5,
                        stop="idempotency")
        return dict(kind=kind, n=_log(rng, 1000, 4096), gap=rng.choice([0.3, 0.05]), prec="split16",
                    slices=rng.choice([4, 5]), stop="parameterless")
    if kind == "water":
        if rng.random() < 0.25:
            return dict(kind=kind, nmol=_log(rng, 30, 110), tau=rng.choice([1e-6, 1e-5]), prec="fp64",
                        trunc=rng.choice(["frobenius", "frobinf"]), part=1024, out="dense")
        nmol = _log(rng, 50, 3500)
        return dict(kind=kind, nmol=nmol, tau=1e-5 if nmol > 1200 else rng.choice([1e-6, 1e-5]), prec="split16",
                    trunc=rng.choice(["frobenius", "frobenius", "frobinf", "mixed"]), part=rng.choice([1024, 4096]),
                    out="host" if nmol < 200 else "tiles")
    if kind == "twopass":
        return dict(kind=kind, nmol=_log(rng, 80, 500), tau=rng.choice([1e-6, 1e-5]), tau1=1e-5)
    if kind == "helix":
        if rng.random() < 0.3:
            return dict(kind=kind, nres=rng.randint(12, 32), tau=1e-6, prec="fp64", autograd=True)
        nres = _log(rng, 40, 1000)
        return dict(kind=kind, nres=nres, tau=rng.choice([1e-6, 1e-5]), prec="split16",
                    autograd=nres < 100 and rng.random() < 0.5)
    return dict(kind=kind, nb=_log(rng, 24, 600), tau=rng.choice([1e-2, 1e-3, 1e-1]),
                trunc=rng.choice(["frobenius", "frobinf"]), part=rng.choice([1024, 4096]))


# ------------------------------------------------------------------ the inputs
class Tiles:
    """A tile set as the entry points take it (n, brow, bcol, val)."""

    def __init__(self, n, brow, bcol, val):
        self.n, self.brow, self.bcol, self.val = n, brow, bcol, val


def _normal(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda", dtype=torch.float64)


def _uniform(g, lo, hi, *shape):
    return lo + (hi - lo) * torch.rand(*shape, generator=g, device="cuda", dtype=torch.float64)


def _dense(n, gap, g):
    """Q diag(lam) Q^T with n/2 eigenvalues on either side of the gap."""
    nocc = n // 2
    q, _ = torch.linalg.qr(_normal(g, n, n))
    occ = _uniform(g, -2.0, -gap / 2, nocc)
    virt = _uniform(g, gap / 2, 2.5 + gap / 2, n - nocc)
    f = (q * torch.cat([occ, virt])) @ q.T
    return 0.5 * (f + f.T), nocc, float(occ.max()), float(virt.min())


def _blocks(m, nbf, g):
    """m symmetric nbf x nbf blocks Q diag(occupied, virtual) Q^T, and the edges of their spectra."""
    q = torch.eye(nbf, device="cuda", dtype=torch.float64).repeat(m, 1, 1)
    for v in _normal(g, nbf, m, nbf):       # nbf random reflections
        v = v / v.norm(dim=1, keepdim=True)
        q -= 2.0 * (q @ v[:, :, None]) * v[:, None, :]
    occ = _uniform(g, -1.5, -0.5, m, nbf // 2)
    virt = _uniform(g, 0.5, 2.5, m, nbf - nbf // 2)
    d = (q * torch.cat([occ, virt], 1)[:, None, :]) @ q.transpose(1, 2)
    return 0.5 * (d + d.transpose(1, 2)), occ.max(), virt.min()


def _assemble(pos, nbf, cutoff, decay, g):
    """Tiles of the matrix of blocks: one on the diagonal for each centre, and
    N(0,1) exp(-r / decay) between centres closer than cutoff, scaled so that
    every row's off-block sum is at most 0.25."""
    m = pos.shape[0]
    diag, homo, lumo = _blocks(m, nbf, g)
    pa, pb = [], []
    for s in range(0, m, 2048):
        near = torch.cdist(pos[s:s + 2048], pos, compute_mode="donot_use_mm_for_euclid_dist") < cutoff
        a, b = near.nonzero(as_tuple=True)
        a = a + s
        pa.append(a[a < b])
        pb.append(b[a < b])
    pa, pb = torch.cat(pa), torch.cat(pb)
    r = (pos[pa] - pos[pb]).norm(dim=1)
    blk = _normal(g, pa.numel(), nbf, nbf) * torch.exp(-r / decay)[:, None, None]
    sums = torch.zeros(m, nbf, device="cuda", dtype=torch.float64)
    mag = blk.abs()
    sums.index_put_((pa,), mag.sum(2), accumulate=True)      # in a fixed order, unlike index_add_
    sums.index_put_((pb,), mag.sum(1), accumulate=True)
    del mag
    edge = float(sums.max())
    scale = min(1.0, 0.25 / edge) if edge > 0 else 1.0
    blk *= scale
    n = m * nbf
    nb = (n + B - 1) // B
    cen = torch.arange(m, device="cuda")
    ra, rb = torch.cat([cen, pa]), torch.cat([cen, pb])
    first, last = (cen * nbf) // B, (cen * nbf + nbf - 1) // B
    keys = []
    for di in range(nbf // B + 2):
        for dj in range(nbf // B + 2):
            i, j = first[ra] + di, first[rb] + dj
            ok = (i <= last[ra]) & (j <= last[rb]) & (i <= j)
            keys.append((i * nb + j)[ok])
    keys = torch.unique(torch.cat(keys))
    val = torch.zeros(keys.numel(), B, B, device="cuda", dtype=torch.float64)
    flat, loc = val.view(-1), torch.arange(nbf, device="cuda")

    def put(a, b, x):
        for s in range(0, a.numel(), 20000):
            rr = (a[s:s + 20000] * nbf)[:, None, None] + loc[None, :, None]
            cc = (b[s:s + 20000] * nbf)[:, None, None] + loc[None, None, :]
            rr, cc = torch.broadcast_tensors(rr, cc)
            up = (rr // B) <= (cc // B)
            rr, cc, v = rr[up], cc[up], x[s:s + 20000][up]
            t = torch.searchsorted(keys, (rr // B) * nb + cc // B)
            flat[t * (B * B) + (rr % B) * B + cc % B] = v
            on = (rr // B) == (cc // B)     # a diagonal tile holds both triangles
            rr, cc, v, t = rr[on], cc[on], v[on], t[on]
            flat[t * (B * B) + (cc % B) * B + rr % B] = v

    put(cen, cen, diag)
    put(pa, pb, blk)
    f = Tiles(n, (keys // nb).int(), (keys % nb).int(), val)
    off = edge * scale
    return f, m * (nbf // 2), float(homo) + off, float(lumo) - off


def _water(nmol, g):
    """Molecules uniform in a cube, along a Morton curve."""
    side = (nmol / DENSITY) ** (1.0 / 3.0)
    pos = _uniform(g, 0.0, side, nmol, 3)
    q = (pos / side * 1024.0).floor().clamp(0, 1023).long()
    code = torch.zeros(nmol, device="cuda", dtype=torch.long)
    for bit in range(10):
        for ax in range(3):
            code |= ((q[:, ax] >> bit) & 1) << (3 * bit + ax)
    return _assemble(pos[torch.argsort(code, stable=True)], WATER, 10.0, 2.0, g)


def _helix(nres, g):
    pos = torch.zeros(nres, 3, device="cuda", dtype=torch.float64)
    pos[:, 0] = 1.5 * torch.arange(nres, device="cuda")
    return _assemble(pos, HELIX, 15.0, 3.0, g)


def _weight(f, g):
    """A symmetric N(0,1) matrix on the tile pattern of f."""
    w = _normal(g, *f.val.shape)
    on = f.brow == f.bcol
    w[on] = 0.5 * (w[on] + w[on].transpose(1, 2))
    pad = -f.n % B
    if pad:
        last = int(f.bcol.max())
        w[f.bcol == last, :, B - pad:] = 0.0
        w[f.brow == last, B - pad:, :] = 0.0
    return Tiles(f.n, f.brow, f.bcol, w)


def _to_dense(f):
    nb = (f.n + B - 1) // B
    a = torch.zeros(nb, nb, B, B, device="cuda", dtype=torch.float64)
    i, j = f.brow.long(), f.bcol.long()
    a[j, i] = f.val.transpose(1, 2)
    a[i, j] = f.val
    return a.permute(0, 2, 1, 3).reshape(nb * B, nb * B)[: f.n, : f.n].contiguous()


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _filled(nb, g):
    """Every upper tile of nb tile rows, norms decaying from the diagonal (a filled-in iterate)."""
    i, j = torch.triu_indices(nb, nb, device="cuda")
    size = torch.exp(-(j - i).double() / 8.0 + 2.0 * _normal(g, i.numel()))
    return Tiles(nb * B, i.int(), j.int(), _normal(g, i.numel(), B, B) * (size / B)[:, None, None])


# ------------------------------------------------------------------ the passes
def prepare(case, seed):
    g = _gen(seed)
    k = case["kind"]
    s = dict(case=case)
    if k == "truncate":
        s["F"] = _filled(case["nb"], g)
        return s
    if k == "dense":
        s["F"], s["nocc"], s["homo"], s["lumo"] = _dense(case["n"], case["gap"], g)
        s["params"] = dict(precision=case["prec"], stop=case["stop"])
        if case["slices"]:
            s["params"]["slices"] = case["slices"]
        return s
    if k == "helix":
        s["F"], s["nocc"], s["homo"], s["lumo"] = _helix(case["nres"], g)
        s["W"] = _weight(s["F"], g)
        s["params"] = dict(precision=case["prec"])
        if case["autograd"]:     # the loss reads W's tile at each of D's tiles
            nb = (s["F"].n + B - 1) // B
            s["Wt"] = torch.zeros(nb, nb, B, B, device="cuda", dtype=torch.float64)
            s["Wt"][s["W"].brow.long(), s["W"].bcol.long()] = s["W"].val
            s["F"].val.requires_grad_(True)
        else:
            s["params"]["record_masks"] = 1
            s["D"] = _buffers(_interp(case["nres"], _HD_TILES), device="cuda")
        return s
    f, s["nocc"], s["homo"], s["lumo"] = _water(case["nmol"], g)
    if k == "twopass":
        s["F"] = _to_dense(f)
        return s
    s["F"] = f
    s["params"] = dict(precision=case["prec"], trunc=case["trunc"], frobinf_part=case["part"])
    most = _interp(case["nmol"], _D_TILES[case["tau"]])
    if case["out"] == "tiles":
        s["D"] = _buffers(most, device="cuda")
    if case["out"] == "host":
        s["F"] = Tiles(f.n, f.brow.cpu().numpy(), f.bcol.cpu().numpy(), f.val.cpu().numpy())
        s["D"] = _buffers(most, pin_memory=True)
    return s


def _buffers(tiles, **where):
    """Room for 1.5 times the usual number of D's tiles."""
    cap = int(1.5 * tiles) + 64
    return (torch.zeros(cap, dtype=torch.int32, **where), torch.zeros(cap, dtype=torch.int32, **where),
            torch.zeros(cap, B, B, dtype=torch.float64, **where))


def _take(ctx, d):
    """D's tiles into the caller's device buffers, through the C entry point."""
    n = ctypes.c_int64()
    rc = sp2.load().sp2_copy_D(ctx.ctx, d[0].data_ptr(), d[1].data_ptr(), d[2].data_ptr(), d[0].numel(), 1,
                               ctypes.byref(n))
    if rc != sp2.SP2_OK:
        raise sp2.SP2Error(rc, "sp2_copy_D")
    return {"brow": d[0], "bcol": d[1], "val": d[2], "tiles": n.value}


def run(s):
    c = s["case"]
    k = c["kind"]
    if k == "dense":
        d, st = sp2.run(s["F"], s["nocc"], s["homo"], s["lumo"], 0.0, **s["params"])
        return {"D": d, "n": st["n"], "triplets": st["tile_triplets"]}
    if k == "truncate":
        return {"keep": sp2.sp2_truncate(s["F"], c["tau"], c["trunc"], c["part"])}
    if k == "twopass":
        d, st, st1, bounds = sp2.run_two_pass(s["F"], s["nocc"], c["tau1"], c["tau"], precision="split16")
        return {"D": d, "n": st["n"], "n1": st1["n"], "bounds": torch.tensor(bounds)}
    f = s["F"]
    if k == "helix" and c["autograd"]:
        f.val.grad = None
        val, brow, bcol = sp2.SP2Function.apply(f.val, f.brow, f.bcol, f.n, s["nocc"], s["homo"], s["lumo"], c["tau"],
                                                s["params"])
        i, j = brow.long(), bcol.long()
        twice = torch.where(brow == bcol, 1.0, 2.0).double()     # a stored tile stands for both triangles
        (val * s["Wt"][i, j]).sum(dim=(1, 2)).mul(twice).sum().backward()
        d = torch.zeros_like(s["Wt"])
        d[i, j] = val.detach()
        return {"D": d, "dF": f.val.grad}
    ctx = sp2.SP2(f, s["nocc"], s["homo"], s["lumo"], c["tau"], **s["params"])
    st = ctx.run()
    out = {"n": st["n"], "triplets": st["tile_triplets"]}
    if k == "water" and c["out"] == "dense":
        out["D"] = ctx.D_dense(device=True)
    elif k == "water" and c["out"] == "host":
        ctx.D_host(s["D"])
        out.update(brow=s["D"][0], bcol=s["D"][1], val=s["D"][2], tiles=st["nnzb_final"])
    else:
        out.update(_take(ctx, s["D"]))
    if k == "helix":
        out["dF"] = ctx.backward(s["W"])[2]
    ctx.close()
    return out


# ------------------------------------------------------------------ what a pass cannot do without
def _interp(x, table):
    xs, ys = [math.log(a) for a, _ in table], [math.log(b) for _, b in table]
    i = 0
    while i + 2 < len(xs) and math.log(x) > xs[i + 1]:
        i += 1
    t = (math.log(x) - xs[i]) / (xs[i + 1] - xs[i])
    return math.exp(ys[i] + t * (ys[i + 1] - ys[i]))


# (molecules or residues, value): stored tiles of F and D and tile-product flops
# of one run, counted on one matrix of the recipe each
_F_TILES = [(30, 275), (101, 2261), (400, 14042), (1000, 41203), (4000, 195839)]
_D_TILES = {1e-6: [(30, 276), (101, 2821), (400, 29974), (1000, 111902), (2000, 295463)],
            1e-5: [(30, 275), (101, 2363), (400, 19134), (1000, 69255), (4000, 453261)]}
_W_FLOPS = {1e-6: [(30, 7.06e9), (101, 2.21e11), (400, 6.54e12), (1000, 3.79e13), (2000, 1.34e14)],
            1e-5: [(30, 7.02e9), (101, 1.73e11), (400, 3.10e12), (1000, 1.60e13), (4000, 1.62e14)]}
_HF_TILES = [(12, 288), (32, 1068), (200, 7620), (1000, 38820)]
_HD_TILES = [(12, 300), (32, 1464), (200, 12596), (1000, 68459)]
_H_FLOPS = [(12, 7.9e9), (32, 7.06e10), (200, 8.07e11), (1000, 4.68e12)]


def work(case):
    """flops: the tile products of all squares, 2 * 32^3 for each (I <= J, K)
    triplet; where the tile pattern decides their number, the count measured on
    matrices of the recipe.  bytes: F read once, D (and the gradient) written once."""
    k = case["kind"]
    tile = 8.0 * B * B
    if k == "dense":
        nb = (case["n"] + B - 1) // B
        squares = 19 if case["gap"] >= 1.0 else 29
        return {"bytes": 16.0 * case["n"] ** 2, "flops": 2.0 * B ** 3 * nb * nb * (nb + 1) / 2 * squares}
    if k == "truncate":
        f = case["nb"] * (case["nb"] + 1) / 2
        return {"bytes": f * (tile + 12.0), "flops": f * 2.0 * B * B}
    if k == "helix":    # forward, and the two products of every reverse step
        f, d = _interp(case["nres"], _HF_TILES), _interp(case["nres"], _HD_TILES)
        return {"bytes": (3 * f + d) * tile, "flops": 3.0 * _interp(case["nres"], _H_FLOPS)}
    flops = _interp(case["nmol"], _W_FLOPS[case["tau"]])
    if k == "twopass":
        return {"bytes": 16.0 * (WATER * case["nmol"]) ** 2, "flops": 2.0 * flops}
    f, d = _interp(case["nmol"], _F_TILES), _interp(case["nmol"], _D_TILES[case["tau"]])
    return {"bytes": (f + d) * tile, "flops": flops}


def tolerance(case):
    """About four times what was seen: FP64 against the eigendecomposition
    (1.5e-14 at n = 512), the sliced products against the FP64 path or the
    eigendecomposition (four slices: water-like 9.5e-10, helix-like 1.0e-9 with
    the gradient, dense with a narrow gap 2.5e-7; five slices: 4.8e-10 at
    n = 4096).  The bounds of a second run come out of small differences of
    sums, which another rounding moves by 1e-7.  Whole numbers stay the same."""
    k = case["kind"]
    if k == "truncate":
        return "exact"
    if k == "twopass":
        return {"rel": 4e-7, "max": 2e-5, "differ": 0.0}
    if case["prec"] == "fp64":
        return {"rel": 2e-13, "max": 1e-11, "differ": 0.0}
    if k == "dense":
        return {"rel": 1e-6, "max": 6e-6, "differ": 0.0} if case["slices"] == 4 else \
               {"rel": 2e-9, "max": 1e-8, "differ": 0.0}
    return {"rel": 5e-9, "max": 2e-6, "differ": 0.0}


# ------------------------------------------------------------------ the same in 64 bits, by eigendecomposition
def exact(case, seed):
    """D = sum of y_i y_i^T over the occupied eigenvectors, and dL/dF from the
    response of that projector; for the forms whose output does not depend on
    the truncated tile pattern, up to sizes that eigh does quickly."""
    k = case["kind"]
    g = _gen(seed)
    if k == "dense" and case["n"] <= 2048:
        f, nocc, _, _ = _dense(case["n"], case["gap"], g)
        _, y = torch.linalg.eigh(f)
        y = y[:, :nocc]
        return {"D": y @ y.T, "n": None, "triplets": None}
    if k == "water" and case["out"] == "dense":
        f, nocc, _, _ = _water(case["nmol"], g)
        _, y = torch.linalg.eigh(_to_dense(f))
        y = y[:, :nocc]
        return {"D": y @ y.T, "n": None, "triplets": None}
    if k == "helix" and case["nres"] <= 32:
        f, nocc, _, _ = _helix(case["nres"], g)
        w = _to_dense(_weight(f, g))
        lam, y = torch.linalg.eigh(_to_dense(f))
        m = y.T @ w @ y
        den = lam[:, None] - lam[None, :]
        occ = (torch.arange(f.n, device="cuda") < nocc).double()
        df = occ[:, None] - occ[None, :]
        grad = y @ (m * torch.where(df != 0, df / torch.where(df != 0, den, 1.0), 0.0)) @ y.T
        nb = (f.n + B - 1) // B
        p = torch.zeros(nb * B, nb * B, device="cuda", dtype=torch.float64)
        p[: f.n, : f.n] = grad
        t = p.view(nb, B, nb, B).permute(0, 2, 1, 3)[f.brow.long(), f.bcol.long()].clone()
        if case["autograd"]:
            t[f.brow != f.bcol] *= 2.0       # a stored tile stands for both triangles
        return {"D": None, "dF": t} if case["autograd"] else {"dF": t}
    return None
