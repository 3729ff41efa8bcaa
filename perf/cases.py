"""Workloads whose time matters to a user of the far-zone solver, each a call through the
public binding (paper_2501_04684_gb300).

A case is a dict of plain values:
  op        matvec | translate | solve | map | train
  shape     full (every box of a grid^3 cube), sphere, cube, ellipsoid (one-box-thick shells)
            or batch (independent shells of all three kinds in one plan)
  radius    shell radius in boxes (grid edge for shape = full)
  members   scatterers of a batch (1 otherwise)
  nb_lo/hi  basis functions per box, drawn per box in this range
  edge      box edge in wavelengths is 1 / edge (4 is the paper's a; 8 and 256 its low-frequency sizes)
  prec      translation arithmetic, which: part of Z (matvec), nrhs: right-hand sides
  symmetry  1: the symmetry-compressed coupling store
  refine    solve: outer refinement around inner GMRES in `inner`
  shuffle   box order: 1 arbitrary, 0 lattice order
Mapping matrices and inputs (and the arbitrary box orders) are drawn from the seed; plans, loaded network weights
and output buffers are what a program keeps between calls.
"""
import math

import numpy as np
import torch

import paper_2501_04684_gb300 as ie

K0 = 2.0 * math.pi
ETA0 = 376.730313668
NU = 192
PREC = {name: p for p, name in ie.PREC_NAMES.items()}
WHICH = {"far": ie.IE_FAR, "near": ie.IE_NEAR, "full": ie.IE_FULL}
BASE = dict(op="matvec", shape="sphere", radius=7.0, members=1, nb_lo=32, nb_hi=32, edge=4, prec="fp16x3", which="full",
            nrhs=1, symmetry=1, refine=0, inner="fp16x3", tol=1e-5, functions=0, steps=0, shuffle=0)


def listed():
    def case(name, **kw):
        return {"name": name, **BASE, **kw}
    return [
        # the smallest product a solver makes: 64 boxes, where launches and latency count
        case("tiny_full_fp32", shape="full", radius=4.0, prec="fp32", symmetry=0),
        # a small request of a serving loop: about 200 boxes, three incidences, GMRES to 1e-5
        case("serve200_solve", op="solve", radius=2.8, nrhs=3),
        # the plain path on the 16^3 shell: one operator application in FP32
        case("shell16_full_fp32", prec="fp32", symmetry=0),
        # the paper's low-frequency box edge, two right-hand sides, one block per displacement
        case("shell16_lfb256_full", edge=256, nrhs=2, symmetry=0),
        # the plain solve of the 16^3 shell to 1e-6
        case("shell16_solve_fp32", op="solve", prec="fp32", inner="fp32", tol=1e-6, symmetry=0),
        # the far product of the 32^3 shell (24.9 M far pairs), the headline operator
        case("shell32_far_fp16x3", radius=14.0, which="far"),
        # the headline solve: FP64 refinement around FP16X3 GMRES on the 32^3 shell
        case("shell32_solve_refined", op="solve", radius=14.0, refine=1),
        # uneven scatterers, box and right-hand-side counts in one plan
        case("batch_full_bf16x3", shape="batch", radius=6.0, members=8, nb_lo=16, nb_hi=64, prec="bf16x3", nrhs=4),
        # the translation stage alone, single-product form, ragged right-hand sides
        case("shell10_translate_fp16x1", op="translate", radius=4.3, prec="fp16x1", nrhs=3, symmetry=0, shuffle=1),
        # translation networks (loaded weights) on the tensor cores
        case("networks_far", radius=6.0, prec="cvfcnn", which="far"),
        # mapping construction of a scatterer's basis functions, host arrays in and out
        case("map_6000", op="map", functions=6000),
        # the networks' training steps, weights read back
        case("train_networks", op="train", radius=4.3, prec="cvfcnn", steps=40),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    c = dict(BASE)
    c["op"] = rng.choices(["matvec", "solve", "translate", "map", "train"], [46, 24, 14, 8, 8])[0]
    if c["op"] == "map":
        c["functions"] = int(_log(rng, 50, 6000))
        c["edge"] = rng.choice([4, 8, 256])
        return c
    c["radius"] = round(_log(rng, 1.6, 14.0), 2)
    c["shape"] = rng.choices(["sphere", "cube", "ellipsoid", "full"], [5, 2, 2, 1])[0]
    if c["shape"] == "full":
        c["radius"] = float(rng.randint(3, 9))
    lo = rng.randint(1, 40)
    c["nb_lo"], c["nb_hi"] = rng.choice([(32, 32), (16, 64), (lo, lo + rng.randint(0, 40))])
    c["shuffle"] = rng.randint(0, 1)
    if c["op"] == "train":
        c.update(shape="sphere", radius=round(_log(rng, 1.6, 4.3), 2), prec="cvfcnn", steps=rng.randint(8, 40), shuffle=0)
        return c
    if c["op"] == "solve":
        c.update(nb_lo=32, nb_hi=32, nrhs=rng.randint(1, 4))
        form = rng.choice(["fp32", "fp16x3", "refined", "mixed"])
        if form == "fp32":
            c.update(prec="fp32", inner="fp32", tol=1e-6)
        elif form == "refined":
            c.update(refine=1)
        elif form == "mixed":
            c.update(refine=1, inner=rng.choice(["bf16x3", "fp16x1"]))
    else:
        c["prec"] = rng.choice(["fp32", "bf16x3", "fp16x3", "fp16x3", "fp16x1", "bf16x1", "cvfcnn"])
        c["which"] = rng.choice(["far", "full", "full", "near"])
        c["nrhs"] = rng.choice([1, 1, 2, 3, 5, 8])
        c["edge"] = rng.choice([4, 4, 4, 8, 256])
        if c["op"] == "matvec" and rng.random() < 0.2:
            c.update(shape="batch", members=rng.randint(2, 10), radius=round(rng.uniform(2.5, 6.0), 2), edge=4, shuffle=0)
    if c["prec"] == "cvfcnn":   # the networks' fit bounds the plan's preparation
        c.update(shape="sphere" if c["shape"] != "batch" else "batch", radius=min(c["radius"], 5.0), edge=4, symmetry=1)
    elif c["shape"] != "full" and c["radius"] <= 7.0:
        c["symmetry"] = rng.randint(0, 1)
    while _cost(c) > 110.0 and (c["nrhs"] > 1 or c["radius"] > 4.0):   # no more than the largest listed case
        if c["nrhs"] > 1:
            c["nrhs"] -= 1
        else:
            c["radius"] = round(0.9 * c["radius"], 2) if c["shape"] != "full" else c["radius"] - 1.0
    return c


def _cost(c):
    """Far pairs x columns, weighted by the arithmetic, in units of about a millisecond."""
    n = _boxes(c, 0)[0].shape[0]
    pairs = n * n / c["members"] * c["nrhs"]
    per = {"fp32": 6.5e-6, "cvfcnn": 1e-6}.get(c["prec"], 0.9e-6)
    return pairs * per * (14 if c["op"] == "solve" else 1)


# ---------------------------------------------------------------- geometry and inputs
def _shell(kind, radius, semi=(1.0, 1.0, 1.0)):
    """Boxes (ijk >= 0) within one box of a sphere / cube / ellipsoid surface, and the grid edge."""
    G = 2 * int(math.ceil(radius + 1.0))
    c = np.stack(np.meshgrid(*[np.arange(G)] * 3, indexing="ij"), -1).reshape(-1, 3)
    x = c + 0.5 - G / 2.0
    if kind == "full":
        g = int(radius)
        return np.stack(np.meshgrid(*[np.arange(g)] * 3, indexing="ij"), -1).reshape(-1, 3).astype(np.int32), g
    if kind == "sphere":
        keep = np.abs(np.sqrt((x * x).sum(1)) - radius) <= 1.0
    elif kind == "cube":
        keep = np.abs(np.abs(x).max(1) - radius) <= 1.0
    else:
        s = radius * np.asarray(semi)
        rho = np.maximum(np.sqrt(((x / s) ** 2).sum(1)), 1e-12)
        grad = np.maximum(np.sqrt(((x / s ** 2) ** 2).sum(1)) / rho, 1e-12)
        keep = np.abs((rho - 1.0) / grad) <= 1.0
    return c[keep].astype(np.int32), G


def _boxes(c, seed):
    """(box_ijk, grid edge, scatterer of each box, right-hand sides of each scatterer)."""
    g = np.random.default_rng([seed, 1])
    if c["shape"] != "batch":
        ijk, G = _shell(c["shape"], c["radius"], (1.0, 0.8, 0.6))
        if c["shuffle"]:
            ijk = ijk[g.permutation(len(ijk))]
        return ijk, G, np.zeros(len(ijk), np.int32), [c["nrhs"]]
    # the members' shapes come from the case, so every seed of it is the same work
    gs = np.random.default_rng([c["members"], int(100 * c["radius"])])
    parts, G, nr = [], 0, []
    for m in range(c["members"]):
        kind = ["sphere", "cube", "ellipsoid"][int(gs.integers(0, 3))]
        semi = (1.0, gs.uniform(0.5, 1.0), gs.uniform(0.5, 1.0))
        b, gm = _shell(kind, max(1.6, c["radius"] * gs.uniform(0.4, 1.0)), semi)
        parts.append(b)
        G = max(G, gm)
        nr.append(int(gs.integers(1, c["nrhs"] + 1)) if m else c["nrhs"])
    group = np.concatenate([np.full(len(b), i, np.int32) for i, b in enumerate(parts)])
    return np.concatenate(parts), G, group, nr


def _complex(gen, *shape):
    return torch.view_as_complex(torch.randn(*shape, 2, generator=gen, device="cuda"))


def _alpha(c):
    """Self term above the operator's norm: the measured one of the 16^3 / 32^3 shells at nb = 32."""
    s = (math.sqrt(c["nb_hi"]) + math.sqrt(NU)) / (math.sqrt(32.0) + math.sqrt(NU))
    low = {4: 1.0, 8: 4.1, 256: 1.1e5}[c["edge"]]
    return (9.31e7 if c["radius"] <= 7.0 and c["shape"] == "sphere" else 1.14e8) * s * s * low


def _make(c, seed):
    """Everything drawn for a case: geometry, P (host and device), inputs."""
    gen = torch.Generator("cuda")
    gen.manual_seed(1000003 * c["nrhs"] + seed)
    ijk, G, group, nr = _boxes(c, seed)
    # the counts come from the case, so every seed of it has the same number of unknowns
    nb = np.random.default_rng([c["nb_lo"], c["nb_hi"]]).integers(c["nb_lo"], c["nb_hi"] + 1, len(ijk)).astype(np.int32)
    n = int(nb.sum())
    d = dict(ijk=ijk, G=G, group=group, nr=nr, nb=nb, n=n, P=_complex(gen, n, NU), alpha=_alpha(c), a=1.0 / c["edge"])
    if c["op"] == "translate":
        d["X"] = _complex(gen, c["nrhs"], len(ijk), NU)
    elif c["op"] == "matvec":
        d["c"] = _complex(gen, c["nrhs"], n)
        off = np.concatenate([[0], np.cumsum(nb)])
        for g, q in enumerate(nr):          # columns a scatterer does not have are zero
            b = np.flatnonzero(group == g)
            d["c"][q:, off[b[0]]:off[b[-1] + 1]] = 0
    elif c["op"] == "solve":
        u = torch.rand(c["nrhs"], 2, generator=gen, device="cuda", dtype=torch.float64).cpu().numpy()
        ct, phi = 2 * u[:, 0] - 1, 2 * math.pi * u[:, 1]
        st = np.sqrt(1 - ct * ct)
        d["khat"] = np.stack([st * np.cos(phi), st * np.sin(phi), ct], 1)
        d["pol"] = np.stack([ct * np.cos(phi), ct * np.sin(phi), -st], 1)
    return d


def _weights(nblk, seed, H=50):
    gen = torch.Generator("cuda")
    gen.manual_seed(77 + seed)
    return [w.cpu().numpy() for w in (_complex(gen, nblk, H, NU) / 14, _complex(gen, nblk, H) * 0.3,
                                      _complex(gen, nblk, NU, H) / 3, _complex(gen, nblk, NU) * 0.1)]


def _functions(c, seed):
    """Basis functions made of one to three point dipoles at positions inside their box."""
    g = np.random.default_rng([seed, 3])
    off = np.zeros(c["functions"] + 1, np.int64)
    np.cumsum(g.integers(1, 4, c["functions"]), out=off[1:])
    m, a = int(off[-1]), 1.0 / c["edge"]
    return off, g.uniform(-0.5 * a, 0.5 * a, (m, 3)), g.standard_normal((m, 3)) + 1j * g.standard_normal((m, 3))


def prepare(case, seed):
    c = {**BASE, **case}
    if c["op"] == "map":
        return dict(c=c, fun=_functions(c, seed))
    d = _make(c, seed)
    precs = [PREC[c["prec"]]] + ([PREC[c["inner"]]] if c["op"] == "solve" else [])
    batch = c["shape"] == "batch"
    pr = ie.make_problem(K0, ETA0, d["a"], d["G"], d["ijk"], d["nb"], d["P"].cpu().numpy().astype(np.complex128), d["alpha"],
                         ie.precmask(*precs), c["nrhs"], symmetry=c["symmetry"], box_group=d["group"] if batch else None,
                         group_alpha=np.full(c["members"], d["alpha"]) if batch else None,
                         group_nrhs=np.asarray(d["nr"], np.int32) if batch else None)
    s = dict(c=c, plan=ie.Plan(pr), seed=seed)
    h, R = s["plan"].handle, c["nrhs"]
    if c["op"] == "translate":
        s["X"], s["y"] = d["X"], torch.zeros_like(d["X"])
    elif c["op"] == "matvec":
        s["x"], s["y"] = d["c"], torch.zeros_like(d["c"])
        if c["prec"] == "cvfcnn":
            ie.ie_cvfcnn_set_weights(h, *_weights(int(s["plan"].stats["n_coupling_blocks"]), seed))
    elif c["op"] == "solve":
        s["v"] = torch.zeros((R, d["n"]), dtype=torch.complex64, device="cuda")
        ie.ie_rhs_plane_wave(h, d["khat"], d["pol"], s["v"])
        s["y"] = torch.zeros_like(s["v"])
        if c["refine"]:
            s["opts"] = ie.solve_opts(tol=c["tol"], prec=PREC[c["inner"]], refine=1, refine_prec=PREC[c["prec"]],
                                      inner_tol=5e-6 if c["inner"] == c["prec"] else 1e-3)
        else:
            s["opts"] = ie.solve_opts(tol=c["tol"], prec=PREC[c["prec"]])
    return s


def run(state):
    c = state["c"]
    if c["op"] == "map":
        off, pos, mom = state["fun"]
        P, res = ie.ie_map_basis(K0, ETA0, 1.0 / c["edge"], off, pos, mom, tikhonov=1e-5)
        return {"P": P, "residual": res}
    h = state["plan"].handle
    if c["op"] == "translate":
        ie.ie_translate(h, PREC[c["prec"]], state["X"], state["y"], c["nrhs"])
        return state["y"]
    if c["op"] == "matvec":
        ie.ie_matvec(h, WHICH[c["which"]], PREC[c["prec"]], state["x"], state["y"], c["nrhs"])
        return state["y"]
    if c["op"] == "solve":
        ie.ie_solve(h, state["v"], state["y"], c["nrhs"], state["opts"])
        return state["y"]
    ie.ie_cvfcnn_train(h, ie.cvfcnn_train_opts(max_steps=c["steps"], eval_every=0, tol=1e-9, seed=state["seed"]))
    return dict(zip(("W1", "b1", "W2", "b2"), ie.ie_cvfcnn_get_weights(h)))


# ---------------------------------------------------------------- what a pass cannot do without
def work(case):
    c = {**BASE, **case}
    if c["op"] == "map":
        n = c["functions"]
        return {"bytes": n * (2 * 72 + NU * 16 + 8), "flops": n * 2 * 8.0 * 384 * NU}
    ijk, G, group, nr = _boxes(c, 0)
    n = int(len(ijk) * (c["nb_lo"] + c["nb_hi"]) / 2)
    far = near = 0          # (pair, right-hand side) columns; stored near pairs
    conv, disp = 0.0, set()
    for g, q in enumerate(nr):
        b = ijk[group == g]
        E = b.max(0) - b.min(0) + 1
        grid = np.zeros(2 * E)
        grid[tuple((b - b.min(0)).T)] = 1
        auto = np.rint(np.fft.ifftn(np.abs(np.fft.fftn(grid)) ** 2).real).astype(np.int64)
        d = np.argwhere(auto > 0)
        cnt = auto[tuple(d.T)]
        d = np.where(d >= E, d - 2 * E, d)
        fz = np.abs(d).max(1) >= 2
        far += int(cnt[fz].sum()) * q
        near += int(cnt[~fz].sum())
        disp |= set(map(tuple, np.sort(np.abs(d[fz]), 1)))
        N = float(np.prod(8.0 * E))
        conv += q * min(6 * 5 * N * math.log2(N), 8.0 * NU * NU * int(cnt[fz].sum()))
    nb2, hid = ((c["nb_lo"] + c["nb_hi"]) / 2) ** 2, 50
    if c["op"] == "train":
        # inputs are generated; weights written once; forward and two backward products per step
        return {"bytes": len(disp) * (2 * NU * hid + NU + hid) * 8.0,
                "flops": len(disp) * c["steps"] * 128.0 * 2 * NU * hid * 8 * 3}
    # The far field of dipoles on one lattice is a discrete convolution: its transforms' work, or
    # the pairs' products where there are few; a network per pair is nonlinear and needs every pair.
    net = c["prec"] == "cvfcnn"
    w = {"bytes": 2 * 8.0 * c["nrhs"] * (len(ijk) * NU if c["op"] == "translate" else n), "flops": 0.0}
    if c["op"] == "translate" or c["which"] in ("far", "full"):
        w["bytes"] += len(disp) * 2.0 * NU * hid * 4 if net else 0.0
        w["flops"] += far * 2.0 * NU * hid * 8 if net else conv
    if c["op"] != "translate" and c["which"] in ("far", "full"):    # the mapping matrices, read once
        w["bytes"] += n * NU * 8.0
        w["flops"] += 2 * 8.0 * n * NU * c["nrhs"]
    if c["op"] != "translate" and c["which"] in ("near", "full"):   # the stored near blocks
        w["bytes"] += near * nb2 * 8.0
        w["flops"] += near * nb2 * 8.0 * c["nrhs"]
    if c["op"] == "solve":      # seven operator applications reach these tolerances
        w = {k: 7.0 * v for k, v in w.items()}
    return w


# ---------------------------------------------------------------- 64-bit values
class _Field:
    """Fields of the boxes' dipoles in 64 bits: the dyadic Green's function summed over the
    common dipole lattice of one scatterer (a discrete convolution), near boxes subtracted."""

    def __init__(self, ijk, a):
        self.ijk = ijk = torch.as_tensor(ijk - ijk.min(0), device="cuda", dtype=torch.int64)
        self.h, self.L = a / 4, [int(8 * (v + 1)) for v in ijk.amax(0)]
        m = [torch.fft.fftfreq(L, 1.0 / L, device="cuda", dtype=torch.float64) for L in self.L]
        self.K = self._dyad(m[0][:, None, None], m[1][None, :, None], m[2][None, None, :])
        self.K = {q: torch.fft.fftn(v) for q, v in self.K.items()}
        s = torch.arange(64, device="cuda")
        self.site = torch.stack([s & 3, (s >> 2) & 3, s >> 4], -1)
        at = 4 * ijk[:, None, :] + self.site
        self.at = (at[..., 0], at[..., 1], at[..., 2])

    def _dyad(self, mx, my, mz):
        r2 = mx * mx + my * my + mz * mz
        here = r2 == 0
        r = torch.sqrt(torch.where(here, torch.ones_like(r2), r2))
        kr = K0 * self.h * r
        psi = -1j * K0 * ETA0 * torch.exp(-1j * kr) / (4 * math.pi * self.h * r) * (~here)
        u, v = 1 - 1j / kr - 1 / kr ** 2, 1 - 3j / kr - 3 / kr ** 2
        q = (mx, my, mz)
        return {(i, j): psi * ((u if i == j else 0) - q[i] / r * (q[j] / r) * v) for i in range(3) for j in range(i, 3)}

    def all(self, x):
        """x (boxes, 192) complex128 -> the field of every other dipole of the scatterer."""
        X = torch.zeros(3, *self.L, dtype=torch.complex128, device="cuda")
        for i in range(3):
            X[(i, *self.at)] = x.reshape(-1, 64, 3)[:, :, i]
            X[i] = torch.fft.fftn(X[i])
        y = torch.empty_like(x).reshape(-1, 64, 3)
        for i in range(3):
            y[:, :, i] = torch.fft.ifftn(sum(self.K[min(i, j), max(i, j)] * X[j] for j in range(3)))[self.at]
        return y.reshape(-1, NU)

    def near(self, x):
        """The part of all() that comes from boxes within Chebyshev distance one."""
        slot = torch.full([int(v) + 3 for v in self.ijk.amax(0)], -1, device="cuda", dtype=torch.int64)
        slot[tuple((self.ijk + 1).T)] = torch.arange(len(self.ijk), device="cuda")
        y = torch.zeros_like(x)
        for d in np.ndindex(3, 3, 3):
            d = torch.tensor(d, device="cuda") - 1
            b = slot[tuple((self.ijk - d + 1).T)]
            t = torch.nonzero(b >= 0)[:, 0]
            m = (4 * d + self.site[:, None, :] - self.site[None, :, :]).double()
            D = self._dyad(m[..., 0], m[..., 1], m[..., 2])
            G = torch.stack([torch.stack([D[min(i, j), max(i, j)] for j in range(3)], -1) for i in range(3)], -1)
            G = G.permute(0, 3, 1, 2).reshape(NU, NU)      # [site, component][site, component]
            y[t] += x[b[t]] @ G.T
        return y


class _Mapped:
    """One scatterer's operator on basis coefficients, 64 bits."""

    def __init__(self, d, g):
        b = np.flatnonzero(d["group"] == g)
        off = np.concatenate([[0], np.cumsum(d["nb"])])
        self.rows = slice(int(off[b[0]]), int(off[b[-1] + 1]))
        self.P = d["P"][self.rows].to(torch.complex128)
        self.box = torch.repeat_interleave(torch.arange(len(b), device="cuda"), torch.as_tensor(d["nb"][b].astype(np.int64), device="cuda"))
        self.nbox, self.alpha, self.field = len(b), d["alpha"], _Field(d["ijk"][b], d["a"])

    def up(self, c):
        return torch.zeros(self.nbox, NU, dtype=torch.complex128, device="cuda").index_add_(0, self.box, self.P * c[:, None])

    def down(self, y):
        return (self.P * y[self.box]).sum(1)

    def apply(self, which, c):
        x = self.up(c)
        f = self.field.near(x) if which == "near" else self.field.all(x)
        if which == "far":
            return self.down(f - self.field.near(x))
        return self.down(f) + self.alpha * c

    def solve(self, v):
        """GMRES in 64 bits to 1e-13."""
        V, H = [v / v.norm()], np.zeros((81, 80), np.complex128)
        for j in range(80):
            w = self.apply("full", V[j])
            for _ in range(2):
                for i, u in enumerate(V):
                    t = torch.vdot(u, w)
                    H[i, j] += complex(t)
                    w = w - t * u
            H[j + 1, j] = float(w.norm())
            e = np.zeros(j + 2, np.complex128)
            e[0] = float(v.norm())
            y, res = np.linalg.lstsq(H[:j + 2, :j + 1], e, rcond=None)[:2]
            if (len(res) and math.sqrt(abs(res[0])) <= 1e-13 * float(v.norm())) or j == 79:
                return sum(complex(q) * u for q, u in zip(y, V))
            V.append(w / w.norm())


def _networks(c, d, seed):
    """Networks of the canonical displacements applied in the frame of every displacement."""
    ijk = torch.as_tensor(d["ijk"], device="cuda", dtype=torch.int64)
    t, b = torch.nonzero((ijk[:, None] - ijk[None, :]).abs().amax(-1) >= 2, as_tuple=True)
    diff = ijk[t] - ijk[b]                             # target - source
    ds, which, count = torch.unique(diff, dim=0, return_inverse=True, return_counts=True)
    order = torch.argsort(which, stable=True)
    t, b = t[order].split(count.tolist()), b[order].split(count.tolist())
    # the library numbers its blocks in the order of their first displacement (lexicographic)
    first = {}
    for v in ds.tolist():
        first.setdefault(tuple(sorted(map(abs, v))), len(first))
    W = [torch.as_tensor(w, device="cuda").to(torch.complex128) for w in _weights(len(first), seed)]
    m = _Mapped(d, 0)
    site = m.field.site
    x = m.up(d["c"][0].to(torch.complex128))
    y, maps = torch.zeros_like(x), {}
    for k, dv in enumerate(ds.tolist()):
        # d = Q c with (Q c)_i = s_i c_p(i): stable order of |d|, no sign on zeros
        order = sorted(range(3), key=lambda i: abs(dv[i]))
        p, s, blk = [order.index(i) for i in range(3)], [-1 if v < 0 else 1 for v in dv], first[tuple(sorted(map(abs, dv)))]
        if (tuple(p), tuple(s)) not in maps:
            l2 = [site[:, p[i]] if s[i] > 0 else 3 - site[:, p[i]] for i in range(3)]
            U = torch.empty(64, 3, dtype=torch.int64, device="cuda")
            sg = torch.empty(64, 3, dtype=torch.float64, device="cuda")
            for i in range(3):
                U[:, p[i]] = 3 * (l2[0] + 4 * l2[1] + 16 * l2[2]) + i
                sg[:, p[i]] = s[i]
            maps[tuple(p), tuple(s)] = U.reshape(-1), sg.reshape(-1)
        U, sg = maps[tuple(p), tuple(s)]
        z = x[b[k]][:, U] * sg
        sc = z.abs().amax(1, keepdim=True)
        hz = (z / sc) @ W[0][blk].T + W[1][blk]
        hz = torch.complex(hz.real.clamp_min(0), hz.imag.clamp_min(0))
        r = torch.empty_like(z)
        r[:, U] = sc * (hz @ W[2][blk].T + W[3][blk]) * sg
        y[t[k]] += r                                   # a displacement's targets are distinct
    return m.down(y)[None]


def _map_exact(c, seed):
    off, pos, mom = _functions(c, seed)
    a, S = 1.0 / c["edge"], 128
    i = np.arange(S)
    ct = 1 - (2 * i + 1) / S
    ph = 2 * np.pi * i / ((1 + math.sqrt(5)) / 2)
    st = np.sqrt(1 - ct * ct)
    smp = 1.5 * a * np.stack([st * np.cos(ph), st * np.sin(ph), ct], 1)

    def fields(at):          # (samples, 3, sources, 3)
        R = smp[:, None] - at[None]
        r = np.linalg.norm(R, axis=-1)
        kr, rh = K0 * r, R / r[..., None]
        psi = -1j * K0 * ETA0 * np.exp(-1j * kr) / (4 * np.pi * r)
        u, v = psi * (1 - 1j / kr - 1 / kr ** 2), psi * (1 - 3j / kr - 3 / kr ** 2)
        D = u[..., None, None] * np.eye(3) - v[..., None, None] * rh[..., :, None] * rh[..., None, :]
        return D.transpose(0, 2, 1, 3)
    s = np.arange(64)
    A = fields(a * ((np.stack([s & 3, (s >> 2) & 3, s >> 4], 1) + 0.5) / 4 - 0.5)).reshape(3 * S, NU)
    B = np.zeros((3 * S, c["functions"]), np.complex128)
    fun = np.repeat(np.arange(c["functions"]), np.diff(off))
    for k in range(0, len(pos), 4096):
        f = np.einsum("lamb,mb->lam", fields(pos[k:k + 4096]), mom[k:k + 4096]).reshape(3 * S, -1)
        np.add.at(B.T, fun[k:k + 4096], f.T)
    aug = np.vstack([A, 1e-5 * np.linalg.norm(A) * np.eye(NU)])
    C = np.linalg.lstsq(aug, np.vstack([B, np.zeros((NU, B.shape[1]))]), rcond=None)[0]
    return {"P": np.ascontiguousarray(C.T), "residual": np.linalg.norm(A @ C - B, axis=0) / np.linalg.norm(B, axis=0)}


def exact(case, seed):
    c = {**BASE, **case}
    if c["op"] == "map":
        return _map_exact(c, seed)
    if c["op"] == "train":
        return None
    d = _make(c, seed)
    if c["op"] == "translate":
        f = _Field(d["ijk"], d["a"])
        X = d["X"].to(torch.complex128)
        if c["prec"] == "cvfcnn":
            return None
        return torch.stack([f.all(x) - f.near(x) for x in X])
    if c["op"] == "matvec" and c["prec"] == "cvfcnn" and c["which"] != "near":
        if c["shape"] == "batch" or c["nrhs"] > 1 or c["which"] != "far":
            return None
        return _networks(c, d, seed)
    y = torch.zeros(c["nrhs"], d["n"], dtype=torch.complex128, device="cuda")
    for g in range(c["members"]):
        m = _Mapped(d, g)
        if c["op"] == "matvec":
            for r in range(d["nr"][g]):
                y[r, m.rows] = m.apply(c["which"], d["c"][r, m.rows].to(torch.complex128))
            continue
        at = torch.as_tensor(d["ijk"], device="cuda").double() + 0.5 - 0.5 * d["G"]
        pos = d["a"] * (at[:, None, :] + (m.field.site.double() + 0.5) / 4 - 0.5)
        for r in range(c["nrhs"]):
            ph = torch.exp(-1j * K0 * (pos @ torch.as_tensor(d["khat"][r], device="cuda")))
            e = ph[..., None] * torch.as_tensor(d["pol"][r], device="cuda")
            y[r] = m.solve(m.down(e.reshape(-1, NU)))
        del m
    return y
