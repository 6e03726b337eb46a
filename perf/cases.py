"""The work a user of this framework has it do, as timed cases.

Twelve cases through the public entry points: batched LLG integration from one
island to the 4096-island census, at both precisions in use; the energy-barrier
band; the surrogate's inference, screening and training; one step of the
kriging optimiser; the assembly of a design's island mesh.  Sizes are those of
the repository's own workloads (bench.py, design.py, model.py, evolve.py) or
lie between them; `draw` spreads them over the same ranges.

`exact` restates every path in FP64 with plain torch and numpy: P1 finite
elements with dense solves, Lindholm's boundary elements, Heun steps, the band
update, the network with autograd, the kriging formulas.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1603_09493_gb300 import _lib as L
from paper_1603_09493_gb300 import api, design_inputs, ego, synth

MU0 = 4e-7 * math.pi
GAMMA_PS = 0.176085963023          # rad / (ps T)
DEV = "cuda"


def listed():
    return [
        # one island of the plain configuration (209 nodes, uniform field), a short run in one call:
        # the smallest LLG call, launches and latency
        dict(name="one island", kind="llg", mesh="small", islands=1, field="uniform", intervals=40,
             precision=L.PREC_BF16X3, one_call=True),
        # one level of the critical-field search of one design: nine fields on the model's own media mesh
        dict(name="field search", kind="llg", mesh="model", islands=9, field="search", intervals=20,
             precision=L.PREC_BF16X3, one_call=True),
        # the labels of a few hundred random designs: a batch over many small meshes, stacked heads
        dict(name="design labels", kind="labels", meshes=12, designs=331, intervals=10),
        # the recording census: thousands of islands on one mesh, advanced and read interval by interval
        dict(name="census", kind="llg", mesh="census", islands=4096, field="head", intervals=1,
             precision=L.PREC_BF16X3, one_call=False),
        # design variants of uneven size with their adjacent-track islands in one batch
        dict(name="uneven variants", kind="uneven", variants=8, realisations=45, intervals=1),
        # the FP32 form of a batch
        dict(name="fp32 batch", kind="llg", mesh="census", islands=200, field="head", intervals=1,
             precision=L.PREC_FP32, one_call=True),
        # energy barriers of the adjacent bits of a few designs on the model's media mesh
        dict(name="barriers", kind="neb", mesh="model", bands=5, images=9, updates=150),
        # surrogate probabilities of a screening population held on the device
        dict(name="surrogate infer", kind="infer", samples=262144),
        # screened error rates of one generation (host arrays, as the design search calls it)
        dict(name="surrogate screen", kind="screen", designs=256, jitter=64),
        # one epoch of training on LLG labels (host arrays, ragged last minibatch)
        dict(name="surrogate train", kind="train", samples=19000, batch=4096),
        # one step of the kriging optimiser: correlation lengths, fit, expected improvement
        dict(name="kriging step", kind="kriging", designs=160, params=12, thetas=32, candidates=4000),
        # the island mesh of one design: operators assembled, exported and released
        dict(name="mesh assembly", kind="mesh", rings=3, slabs=12),
    ]


def _spread(rng, lo, hi):
    """A whole number, uniform in its logarithm."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["llg", "llg", "llg", "labels", "uneven", "neb", "infer", "screen", "train", "kriging", "mesh"])
    if kind == "llg":
        mesh = rng.choice(["small", "model", "census"])
        fp32 = rng.random() < 0.2
        top = (512 if fp32 else 2048) if mesh == "census" else 4096
        B = _spread(rng, 1, top)
        return dict(kind=kind, mesh=mesh, islands=B, field=rng.choice(["uniform", "search", "head"]),
                    intervals=1 if B > 256 else rng.randint(2, 10), precision=L.PREC_FP32 if fp32 else L.PREC_BF16X3,
                    one_call=rng.random() < 0.5)
    if kind == "labels":
        return dict(kind=kind, meshes=rng.randint(2, 16), designs=_spread(rng, 20, 1500), intervals=rng.randint(2, 6))
    if kind == "uneven":
        return dict(kind=kind, variants=rng.randint(2, 8), realisations=_spread(rng, 4, 80), intervals=1)
    if kind == "neb":
        return dict(kind=kind, mesh=rng.choice(["small", "model"]), bands=_spread(rng, 1, 40),
                    images=rng.randint(5, 16), updates=rng.randint(20, 120))
    if kind == "infer":
        return dict(kind=kind, samples=_spread(rng, 100, 262144))
    if kind == "screen":
        return dict(kind=kind, designs=_spread(rng, 10, 1000), jitter=rng.randint(8, 128))
    if kind == "train":
        return dict(kind=kind, samples=_spread(rng, 1000, 32768), batch=rng.choice([1000, 2048, 4096]))
    if kind == "kriging":
        return dict(kind=kind, designs=_spread(rng, 20, 240), params=rng.randint(2, 12), thetas=rng.randint(16, 64),
                    candidates=_spread(rng, 1000, 30000))
    return dict(kind=kind, rings=rng.randint(2, 4), slabs=rng.randint(8, 14))


# --------------------------------------------------------------------------
# inputs, from the seed alone
# --------------------------------------------------------------------------

def _mesh(name):
    """(mesh, materials) of the plain configuration, of the model evaluation's media and of the census."""
    if name == "model":
        return (synth.layered_island_mesh(12.0, 6.0, 6.0, rings=3, hard_slabs=6, soft_slabs=6, seed=7),
                synth.ecc_materials(interlayer_scale=0.2))
    return (synth.small_island_mesh() if name == "small" else synth.census_island_mesh()), synth.ecc_materials()


def _llg(case, seed):
    """Meshes, islands, run parameters and head map of the LLG cases."""
    kind = case["kind"]
    if kind == "labels":
        grid = design_inputs.grid_meshes()
        pick = (np.arange(case["meshes"]) * 37 + 5) % len(grid)
        D = case["designs"]
        Z = synth.counter_uniform(seed, 710, np.arange(D * 12)).reshape(D, 12)
        Zh = synth.counter_uniform(seed, 711, np.arange(8 * 3)).reshape(8, 3)
        R = design_inputs.RANGES
        heads = np.stack([R[k][0] + (R[k][1] - R[k][0]) * Zh[:, j] for j, k in enumerate(design_inputs.HEAD_KEYS)], 1)
        reals = design_inputs.realisations(Z, 1, seed, 0, heads=heads, head_of_design=np.arange(D) % 8)
        # each geometry of the grid goes to one of the picked meshes
        isl = synth.Islands.concat(design_inputs.islands(reals, np.arange(len(grid)) % len(pick), np.arange(D)))
        p = design_inputs.run_params(20.0)
        p.t0_ps = 60.0
        return [grid[i] for i in pick], isl, p, design_inputs.head_stack(heads)
    if kind == "uneven":
        variants = synth.design_variants()[::2][:case["variants"]]
        meshes = [(v["mesh"], synth.ecc_materials()) for v in variants]
        isl, _ = synth.uneven_batch(variants, list(range(len(variants))), case["realisations"], seed=seed,
                                    layout="staggered")
        p = synth.census_run_params()
        p.substeps, p.t0_ps = 0, 50.0
        return meshes, isl, p, synth.synthetic_head_map()
    meshes = [_mesh(case["mesh"])]
    B = case["bands"] if kind == "neb" else case["islands"]
    isl = synth.jittered_islands(B, seed=seed)
    hm = synth.synthetic_head_map()
    if kind == "neb":
        isl.pos_nm[:, 1] += 12.7                    # the adjacent track
        return meshes, isl, synth.RunParams(dt_ps=0.1, rise_ps=0.0, use_map=True, v_m_per_s=0.0, x0_nm=2.0), hm
    p = synth.RunParams(dt_ps=0.1, alpha=0.1, rise_ps=100.0, v_m_per_s=20.0, x0_nm=-2.0, use_map=True, substeps=0,
                        t0_ps=60.0)
    if case["field"] == "uniform":
        p.rise_ps, p.t0_ps, p.use_map, p.uniform_T = 50.0, 30.0, False, synth.uniform_field(1.2, 170.0)
    elif case["field"] == "search":                 # constant fields 0 .. 4 sigma against the head field
        mag = 0.034 * 0.5 * (np.arange(B) % 9)
        isl.Hext_T[:] = (-mag[:, None] * synth.head_field_direction()[None]).astype(np.float32)
    return meshes, isl, p, hm


def _start_state(isl, n, seed):
    """Random states near +z: a tilt per island and a ripple per node."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    B = len(isl.mesh_id)
    m = 0.3 * torch.randn((B, 3, 1), generator=g, device=DEV) + 0.03 * torch.randn((B, 3, n), generator=g, device=DEV)
    m[:, 2] += 1.0
    return (m / m.norm(dim=1, keepdim=True)).contiguous()


SIZES = [16, 256, 256, 256, 256, 2]
TRAIN = dict(lr=1e-3, weight_decay=1e-4)


def _samples(N, seed):
    g = torch.Generator(device=DEV).manual_seed(seed)
    return torch.rand((N, 16), generator=g, device=DEV) * 2 - 1


def _labels(X, seed):
    """Outcomes of a smooth rule with a few wrong ones."""
    g = torch.Generator(device=DEV).manual_seed(seed + 1)
    a = X[:, 0] + 0.7 * X[:, 1] * X[:, 2] - 0.4 * X[:, 3]
    y = torch.stack([a > 0.1, a + X[:, 4] < -0.6], 1)
    return (y ^ (torch.rand(y.shape, generator=g, device=DEV) < 0.02)).float()


def _kriging(case, seed):
    n, d = case["designs"], case["params"]
    X = synth.unit_points(n, d, seed, 0)
    y = np.sin(3.0 * X).sum(1) + 0.3 * synth.counter_normal(seed, 900, np.arange(n))
    draws = [synth.theta_unit_draws(case["thetas"], d, seed, r) for r in range(4)]
    half = case["candidates"] // 2
    return X, y, draws, synth.unit_points(half, d, seed, 1), synth.unit_points(half, d, seed, 2)


def _design_mesh(case, seed):
    hard = case["slabs"] // 2
    mesh = synth.layered_island_mesh(12.0, 6.0, 6.0, rings=case["rings"], hard_slabs=hard,
                                     soft_slabs=case["slabs"] - hard, seed=seed)
    scale = 0.1 + 0.9 * float(synth.counter_uniform(seed, 901, np.arange(1))[0])
    return mesh, synth.ecc_materials(Ms_hard=0.557e6, Ku_hard=0.8e6, Ms_soft=0.557e6, Ku_soft=0.16e6,
                                     interlayer_scale=scale)


# --------------------------------------------------------------------------
# the passes
# --------------------------------------------------------------------------

def prepare(case, seed):
    kind = case["kind"]
    if kind in ("infer", "screen", "train"):
        ctx = api.Context(0)
        w = synth.mlp_init_params(SIZES, seed=seed)
        N = case["designs"] * case["jitter"] if kind == "screen" else case["samples"]
        X = _samples(N, seed)
        s = dict(case=case, ctx=ctx, w=w, X=X if kind == "infer" else X.cpu().numpy())
        if kind == "train":
            s["Y"] = _labels(X, seed).cpu().numpy()
        else:
            s["sur"] = ctx.surrogate((16, 256, 4, 2), w)
        return s
    if kind == "kriging":
        return dict(case=case, ctx=api.Context(0), data=_kriging(case, seed))
    if kind == "mesh":
        return dict(case=case, ctx=api.Context(0), mesh=_design_mesh(case, seed))
    ctx = api.Context(0)
    meshes, isl, p, hm = _llg(case, seed)
    ids = np.array([ctx.mesh_upload(*mm) for mm in meshes], np.int32)
    isl.mesh_id = ids[isl.mesh_id]
    s = dict(case=case, ctx=ctx, isl=isl, p=p, map_id=ctx.headmap_upload(hm))
    if kind == "neb":
        s["step"] = _band_step(meshes[0], isl, *ctx.stable_substeps(isl, p, s["map_id"]))
    elif not case.get("one_call", kind == "labels"):
        n = max(mm[0].n_nodes for mm in meshes)
        s["batch"] = ctx.batch(isl, p, precision=case.get("precision", L.PREC_BF16X3), map_id=s["map_id"])
        m = _start_state(isl, n, seed)
        s["batch"].set_state(m, p.t0_ps)
        B = len(isl.mesh_id)
        s["out"] = dict(m=torch.zeros_like(m), switched=torch.zeros(B, dtype=torch.uint8, device=DEV),
                        t_sw=torch.zeros(B, device=DEV), status=torch.zeros(B, dtype=torch.int32, device=DEV),
                        mz=torch.zeros(B, device=DEV))
    return s


def run(s):
    case, ctx = s["case"], s["ctx"]
    kind = case["kind"]
    if kind == "infer":
        return s["sur"].infer(s["X"])
    if kind == "screen":
        return s["sur"].screen(s["X"], case["designs"], case["jitter"])
    if kind == "train":
        sur = ctx.surrogate((16, 256, 4, 2), s["w"])
        curve = sur.train(s["X"], s["Y"], 1, case["batch"], **TRAIN)
        out = dict(params=sur.params(), loss=curve)
        sur.destroy()
        return out
    if kind == "kriging":
        X, y, draws, far, near = s["data"]
        theta, v = ego.theta_search(ctx, X, y, draws)
        with ego.Kriging(ctx, X, y, theta) as gp:
            yhat, std, ei = gp.predict(ego.search_set(X, y, far, near), float(y.min()))
        return dict(theta=theta, nll=v, yhat=yhat, s=std, ei=ei)
    if kind == "mesh":
        mid = ctx.mesh_upload(*s["mesh"])
        out = dict(demag=ctx.get_operator(mid, L.OP_DEMAG_F32), exchange=ctx.get_operator(mid, L.OP_EXCHANGE_F32),
                   volumes=ctx.get_operator(mid, L.OP_VOLUMES_F64), Ms=ctx.get_operator(mid, L.OP_NODAL_MS_F64),
                   Ku=ctx.get_operator(mid, L.OP_NODAL_KU_F64),
                   lambda_max=ctx.mesh_info(mid)["exchange_lambda_max_T"])
        ctx.mesh_release(mid)
        return out
    if kind == "neb":
        r = ctx.neb(s["isl"], case["images"], case["updates"], s["step"], 1.0, case["updates"] // 3,
                    map_id=s["map_id"], head_x_nm=s["p"].x0_nm, want_path=True)
        # the energies are sums over FP32 fields of an FP32 path
        return dict(m=r["m"], E=r["E"].astype(np.float32))
    if "batch" in s:
        o = s["out"]
        s["batch"].advance(case["intervals"])
        s["batch"].read_device(o["m"], o["switched"], o["t_sw"], o["status"], o["mz"])
        return o
    return ctx.run_batch(s["isl"], s["p"], case["intervals"], precision=case.get("precision", L.PREC_BF16X3),
                         map_id=s["map_id"])


def _products(case):
    """(products of a batch row with its mesh's operator, operator entries, nodes x islands) per demag pass."""
    meshes, isl, p, hm = _llg(case, 1)
    ids = np.asarray(isl.mesh_id)
    n = np.array([mm[0].n_nodes for mm in meshes], np.float64)
    rows = np.bincount(ids, minlength=len(meshes)).astype(np.float64)
    return float((rows * 9 * n * n).sum()), float((9 * n * n).sum()), float((rows * n).sum())


# Heun steps of an interval, about: the step rule's count on these meshes
STEPS = dict(small=8, model=7, census=28, labels=12, uneven=44)


def work(case):
    """Inputs read once and outputs written once; the arithmetic of the matrix products (three BF16
    products per demag product at the split precision) and of the assembly's solves."""
    kind = case["kind"]
    if kind in ("infer", "screen", "train"):
        N = case["designs"] * case["jitter"] if kind == "screen" else case["samples"]
        f = 2.0 * sum(a * b for a, b in zip(SIZES[:-1], SIZES[1:]))
        P = sum(a * b + b for a, b in zip(SIZES[:-1], SIZES[1:]))
        if kind == "train":
            return dict(bytes=N * 72.0 + 2 * 4.0 * P, flops=3.0 * f * N)
        return dict(bytes=N * 64.0 + (8.0 * N if kind == "infer" else 16.0 * case["designs"]), flops=f * N)
    if kind == "kriging":
        n, d, T, N = case["designs"], case["params"], 4 * case["thetas"], case["candidates"]
        return dict(bytes=8.0 * (n * d + T * d + N * (d + 3)), flops=(T + 2) * n ** 3 / 3 + 1.0 * N * n * n + 3.0 * d * n * (N + T * n / 2))
    if kind == "mesh":
        n = (1 + 3 * case["rings"] * (case["rings"] + 1)) * (case["slabs"] + 1)
        return dict(bytes=4.0 * 9 * n * n + 4.0 * n * n, flops=2.0 * (2 * n) ** 2 * 3 * n)
    if kind == "neb":
        pr, op, nodes = _products(case)
        P, U = case["images"], case["updates"]
        return dict(bytes=4 * op + 12 * nodes * P, flops=6 * pr * P * (U + 1))
    pr, op, nodes = _products(case)
    fp32 = case.get("precision") == L.PREC_FP32
    k = STEPS[case["mesh"]] if kind == "llg" else STEPS[kind]
    return dict(bytes=4 * op + 24 * nodes, flops=(2 if fp32 else 6) * pr * 2 * k * case["intervals"])


# --------------------------------------------------------------------------
# the same in 64 bits
# --------------------------------------------------------------------------

def _t(a):
    return torch.as_tensor(np.asarray(a, np.float64), device=DEV)


class _Fem:
    """Dense FP64 operators of one island mesh: volumes, nodal Ms and Ku, the exchange matrix S
    (B_ex = -S m, tesla), the Fredkin-Koehler demag matrix N (H = -N M, rows c n + i)."""

    def __init__(self, mesh, mats):
        xyz, tets = _t(mesh.xyz_nm), torch.as_tensor(np.asarray(mesh.tets, np.int64), device=DEV)
        mat = _t(np.asarray(mats))[torch.as_tensor(np.asarray(mesh.tet_region, np.int64), device=DEV)]
        n = self.n = xyz.shape[0]
        p = xyz[tets]
        J = p[:, 1:] - p[:, :1]
        vol = torch.linalg.det(J).abs() / 6
        g = torch.linalg.inv(J).transpose(1, 2)
        g = torch.cat([-g.sum(1, keepdim=True), g], 1)                       # [nt][4][3] gradients

        def lump(q):
            return torch.zeros(n, dtype=torch.float64, device=DEV).index_add_(0, tets.reshape(-1), q.repeat_interleave(4) / 4)

        def dense(v):                                                        # v [nt][4][4] -> [n][n]
            i, j = tets[:, :, None].expand(-1, 4, 4), tets[:, None, :].expand(-1, 4, 4)
            return torch.zeros((n, n), dtype=torch.float64, device=DEV).index_put_(
                (i.reshape(-1), j.reshape(-1)), v.reshape(-1), accumulate=True)

        V = self.V = lump(vol)
        self.Ms, self.Ku = lump(vol * mat[:, 0]) / V, lump(vol * mat[:, 1]) / V
        stiff = vol[:, None, None] * torch.einsum("tac,tbc->tab", g, g)
        KL, KA = dense(stiff), dense(stiff * mat[:, 2][:, None, None])
        self.S = 2e18 * KA / (self.Ms * V)[:, None]
        sq = torch.sqrt(2e18 / (self.Ms * V))
        self.lam = float(torch.linalg.eigvalsh(sq[:, None] * KA * sq[None])[-1])
        q = vol[:, None, None] / 4
        R = torch.cat([dense((q * g[:, :, c:c + 1]).expand(-1, 4, 4)) for c in range(3)], 1)      # [n][3n]
        grad = [dense((q * g[:, None, :, c]).expand(-1, 4, 4)) / V[:, None] for c in range(3)]
        u1 = torch.linalg.solve(KL + 1.0 / n, R)
        u1 = u1 - u1.mean(0, keepdim=True)
        nodes, D = self._boundary(xyz, tets)
        inner = torch.ones(n, dtype=torch.bool, device=DEV)
        inner[nodes] = False
        u = u1.clone()
        u2 = D @ u1[nodes]
        u[nodes] += u2
        if bool(inner.any()):
            u[inner] -= torch.linalg.solve(KL[inner][:, inner], KL[inner][:, nodes] @ u2)
        self.N = torch.cat([G @ u for G in grad], 0)
        self.xyz, self.w = xyz, V / V.sum()

    @staticmethod
    def _solid(a, b, c):
        la, lb, lc = a.norm(dim=-1), b.norm(dim=-1), c.norm(dim=-1)
        num = (a * torch.linalg.cross(b, c)).sum(-1)
        return 2 * torch.atan2(num, la * lb * lc + (a * b).sum(-1) * lc + (a * c).sum(-1) * lb + (b * c).sum(-1) * la)

    def _boundary(self, xyz, tets):
        """Boundary nodes and the matrix from u1 to u2 on them (Lindholm's weights, interior angles)."""
        f = torch.cat([tets[:, [1, 2, 3]], tets[:, [0, 2, 3]], tets[:, [0, 1, 3]], tets[:, [0, 1, 2]]])
        opp = torch.cat([tets[:, k] for k in range(4)])
        _, inv, cnt = torch.unique(f.sort(1).values, dim=0, return_inverse=True, return_counts=True)
        f, opp = f[cnt[inv] == 1], opp[cnt[inv] == 1]
        y = xyz[f]
        out = (torch.linalg.cross(y[:, 1] - y[:, 0], y[:, 2] - y[:, 0]) * (xyz[opp] - y[:, 0])).sum(-1) > 0
        f = torch.where(out[:, None], f[:, [0, 2, 1]], f)
        nodes = torch.unique(f)
        nb = nodes.numel()
        at = torch.zeros(xyz.shape[0], dtype=torch.long, device=DEV)
        at[nodes] = torch.arange(nb, device=DEV)
        omega = torch.zeros(xyz.shape[0], dtype=torch.float64, device=DEV)
        for a in range(4):
            r = [xyz[tets[:, b]] - xyz[tets[:, a]] for b in range(4) if b != a]
            omega.index_add_(0, tets[:, a], self._solid(*r).abs())
        D = torch.diag(omega[nodes] / (4 * math.pi) - 1)
        y = xyz[f]
        e = y.roll(-1, 1) - y
        ln = e.norm(dim=-1)
        xi = e / ln[..., None]
        cr = torch.linalg.cross(y[:, 1] - y[:, 0], y[:, 2] - y[:, 0])
        area2 = cr.norm(dim=-1)
        nrm = cr / area2[:, None]
        gam = torch.einsum("fki,fji->fkj", xi, xi)
        side = torch.linalg.cross(nrm[:, None].expand_as(xi), xi)
        for lo in range(0, nb, 256):
            x = xyz[nodes[lo:lo + 256]]
            rho = y[None] - x[:, None, None]                                 # [b][f][3][3]
            zeta = (nrm[None] * rho[:, :, 0]).sum(-1)
            eta = (side[None] * rho).sum(-1)
            lr = rho.norm(dim=-1)
            ls = lr + lr.roll(-1, 2)
            own = (f[None] == nodes[lo:lo + 256, None, None]).any(-1)       # the observer lies in the face's plane
            P = torch.log((ls + ln[None]) / torch.where(own[..., None], torch.ones_like(ls), ls - ln[None]))
            om = self._solid(rho[:, :, 0], rho[:, :, 1], rho[:, :, 2])
            gp = torch.einsum("fkj,bfj->bfk", gam, P)
            w = (ln / area2[:, None])[None] * (-eta * om[..., None] + zeta[..., None] * gp)
            w = torch.where(own[..., None], torch.zeros_like(w), w.roll(-1, 2))
            for k in range(3):
                D[lo:lo + 256].index_add_(1, at[f[:, k]], -w[:, :, k] / (4 * math.pi))
        return nodes, D


class _Field:
    """FP64 effective field of the islands of one mesh; states are [b][3][n]."""

    def __init__(self, fem, isl, rows, p, hm):
        self.f, self.p, self.hm = fem, p, hm if p.use_map else None
        g = lambda a: _t(np.asarray(a, np.float32)[rows])
        self.ms, self.ku, self.u, self.pos, self.hext = (g(isl.Ms_scale), g(isl.Ku_scale), g(isl.u), g(isl.pos_nm),
                                                         g(isl.Hext_T))
        self.msn = self.ms[:, None] * fem.Ms[None]
        self.NT, self.ST = fem.N.T.contiguous(), fem.S.T.contiguous()
        if self.hm is not None:
            self.B = _t(hm.B_T).reshape(-1, 3)
            self.org, self.h = [float(v) for v in np.float32(hm.origin_nm)], float(np.float32(hm.h_nm))
            self.dim = hm.B_T.shape[:3]

    def head(self, xh):
        f, lo, fr = self.f, [], []
        for c, shift in ((0, self.pos[:, :1] - xh), (1, self.pos[:, 1:]), (2, 0 * self.pos[:, :1])):
            top = self.dim[2 - c]
            v = ((f.xyz[None, :, c] + shift - self.org[c]) / self.h).clamp(0, top - 1)
            i = v.floor().clamp(max=top - 2)
            lo.append(i.long())
            fr.append(v - i)
        out = 0
        for dz in (0, 1):
            for dy in (0, 1):
                for dx in (0, 1):
                    w = (fr[0] if dx else 1 - fr[0]) * (fr[1] if dy else 1 - fr[1]) * (fr[2] if dz else 1 - fr[2])
                    at = ((lo[2] + dz) * self.dim[1] + lo[1] + dy) * self.dim[2] + lo[0] + dx
                    out = out + w[..., None] * self.B[at]
        return out.transpose(1, 2)

    def parts(self, m, ramp, xh):
        """(quadratic terms' field, linear terms' field)."""
        f, (b, _, n) = self.f, m.shape
        q = -(m @ self.ST) / self.ms[:, None, None]
        q += ((2 * f.Ku / f.Ms)[None] * (self.ku / self.ms)[:, None] * torch.einsum("bci,bc->bi", m, self.u))[:, None] * self.u[:, :, None]
        q -= MU0 * ((self.msn[:, None] * m).reshape(b, 3 * n) @ self.NT).reshape(b, 3, n)
        lin = (ramp * _t(self.p.uniform_T)[None] + self.hext)[:, :, None].expand(-1, -1, n)
        return q, lin + ramp * self.head(xh) if self.hm is not None else lin


def _heun(F, m, p, k, intervals):
    h, gp = p.dt_ps / k, GAMMA_PS / (1 + p.alpha ** 2)

    def rhs(m, t):
        q, lin = F.parts(m, min(1.0, t / p.rise_ps) if p.rise_ps > 0 else 1.0, p.x0_nm + p.v_m_per_s * 1e-3 * t)
        c = torch.linalg.cross(m, q + lin, dim=1)
        return -gp * (c + p.alpha * torch.linalg.cross(m, c, dim=1))

    unit = lambda v: v / v.norm(dim=1, keepdim=True)
    mean = lambda m: m[:, 2] @ F.f.w
    z = mean(m)
    t_sw = torch.where(z <= 0, p.t0_ps, -1.0).double()
    for s in range(intervals * k):
        t = p.t0_ps + s * h
        k1 = rhs(m, t)
        m = unit(m + 0.5 * h * (k1 + rhs(unit(m + h * k1), t + h)))
        z, before = mean(m), z
        t_sw = torch.where((t_sw < 0) & (z <= 0), t + h * before / (before - z), t_sw)
    return m, z, t_sw


def _steps(fems, isl, p, hm):
    """Heun steps per interval: the smallest k with gamma/(1+alpha^2) B dt/k <= 1/2, B the largest
    field bound over the meshes."""
    ids, top = np.asarray(isl.mesh_id), 0.0
    for g, f in enumerate(fems):
        r = ids == g
        if not r.any():
            continue
        ms, ku = isl.Ms_scale[r].astype(np.float64), isl.Ku_scale[r].astype(np.float64)
        top = max(top, f.lam / ms.min() + float((2 * f.Ku / f.Ms).max()) * (ku / ms).max()
                  + MU0 * float(f.Ms.max()) * ms.max()
                  + np.linalg.norm(isl.Hext_T[r].astype(np.float64), axis=1).max())
    top += float(np.linalg.norm(np.asarray(p.uniform_T, np.float32).astype(np.float64)))
    if p.use_map:
        top += float(np.linalg.norm(hm.B_T.astype(np.float64), axis=-1).max())
    return max(1, math.ceil(GAMMA_PS / (1 + p.alpha ** 2) * top * p.dt_ps / 0.5)), top


def _band_step(mm, isl, k, bound):
    """Band step from the field bound: step x max Ms x bound = 0.4 (the explicit update's limit)."""
    return 0.4 / (max(float(np.asarray(mm[1])[:, 0].max()), 0.0) * 1e-6 * float(isl.Ms_scale.max()) * bound)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("infer", "screen", "train"):
        return _exact_surrogate(case, seed)
    if kind == "kriging":
        return _exact_kriging(case, seed)
    if kind == "mesh":
        f = _Fem(*_design_mesh(case, seed))
        return dict(demag=-MU0 * 1e6 * f.N, exchange=f.S, volumes=f.V, Ms=f.Ms, Ku=f.Ku, lambda_max=f.lam)
    if work(case)["flops"] / (6 if case.get("precision", 1) else 2) * 2 > 1.2e13:
        return None                                 # over about 20 seconds of FP64 products
    meshes, isl, p, hm = _llg(case, seed)
    fems = [_Fem(*mm) for mm in meshes]
    if kind == "neb":
        return _exact_band(case, fems[0], meshes[0], isl, p, hm)
    k, _ = _steps(fems, isl, p, hm)
    ids, B, n = np.asarray(isl.mesh_id), len(isl.mesh_id), max(f.n for f in fems)
    m = torch.zeros((B, 3, n), dtype=torch.float64, device=DEV)
    z, t_sw = (torch.zeros(B, dtype=torch.float64, device=DEV) for _ in range(2))
    handle = not case.get("one_call", kind == "labels")
    m0 = _start_state(isl, n, seed).double() if handle else None
    for g, f in enumerate(fems):
        rows = np.nonzero(ids == g)[0]
        if rows.size == 0:
            continue
        at = torch.as_tensor(rows, device=DEV)
        if m0 is not None:
            a = m0[at][:, :, :f.n].contiguous()
        else:
            a = torch.zeros((rows.size, 3, f.n), dtype=torch.float64, device=DEV)
            a[:, 2] = 1.0
        a, z[at], t_sw[at] = _heun(_Field(f, isl, rows, p, hm), a, p, k, case["intervals"])
        m[at, :, :f.n] = a
    out = dict(m=m, switched=None, t_sw=t_sw, status=None)
    if handle:
        out["mz"] = z
    return out


def _exact_band(case, f, mm, isl, p, hm):
    D, P, U = case["bands"], case["images"], case["updates"]
    step, spring, climb = _band_step(mm, isl, *_steps([f], isl, p, hm)), 1.0, case["updates"] // 3
    F = _Field(f, isl, np.repeat(np.arange(D), P), p, hm)
    th = math.pi * np.arange(P) / (P - 1)
    m = _t(np.stack([np.sin(th), 0 * th, np.cos(th)], 1))[None, :, :, None].expand(D, P, 3, f.n).contiguous()
    dens = (F.msn * 1e-6).reshape(D, P, 1, f.n)
    dot = lambda a, b: (a * b).sum(2) @ f.w

    def energy(m):
        q, lin = F.parts(m.reshape(D * P, 3, f.n), 1.0, p.x0_nm)
        e = ((0.5 * q + lin) * m.reshape(D * P, 3, f.n)).sum(1) * F.msn
        return -(e @ f.V).reshape(D, P) * 1e-27, (q + lin).reshape(D, P, 3, f.n)

    perp = lambda v, m: v - (v * m).sum(2, keepdim=True) * m
    for it in range(U):
        E, B = energy(m)
        g = dens * perp(B, m)
        up, dn, c = m[:, 2:] - m[:, 1:-1], m[:, 1:-1] - m[:, :-2], m[:, 1:-1]
        Em, E0, Ep = E[:, :-2], E[:, 1:-1], E[:, 2:]
        big, small = torch.maximum((Ep - E0).abs(), (Em - E0).abs()), torch.minimum((Ep - E0).abs(), (Em - E0).abs())
        one, zero = torch.ones_like(E0), torch.zeros_like(E0)
        rising, falling = (Ep > E0) & (E0 > Em), (Ep < E0) & (E0 < Em)
        cp = torch.where(rising, one, torch.where(falling, zero, torch.where(Ep > Em, big, small)))
        cm = torch.where(rising, zero, torch.where(falling, one, torch.where(Ep > Em, small, big)))
        t = perp(cp[..., None, None] * up + cm[..., None, None] * dn, c)
        t = t / dot(t, t).sqrt().clamp(min=1e-300)[..., None, None]
        gt = dot(g[:, 1:-1], t)
        pull = spring * (dot(up, up).sqrt() - dot(dn, dn).sqrt()) - gt
        if it >= climb:
            top = E0.argmax(1, keepdim=True)
            pull = pull.scatter(1, top, -2 * gt.gather(1, top))
        g[:, 1:-1] += pull[..., None, None] * t
        m = m + step * g
        m = m / m.norm(dim=2, keepdim=True)
    return dict(m=m, E=energy(m)[0])


def _exact_surrogate(case, seed):
    N = case["designs"] * case["jitter"] if case["kind"] == "screen" else case["samples"]
    X32 = _samples(N, seed)
    X = X32.double()
    par, off, w = [], 0, synth.mlp_init_params(SIZES, seed=seed)
    for a, b in zip(SIZES[:-1], SIZES[1:]):
        par.append((_t(w[off:off + a * b]).reshape(b, a), _t(w[off + a * b:off + a * b + b])))
        off += a * b + b

    def net(x):
        for i, (W, c) in enumerate(par):
            x = x @ W.T + c
            if i + 1 < len(par):
                x = torch.nn.functional.gelu(x)
        return x

    if case["kind"] == "infer":
        return torch.sigmoid(net(X))
    if case["kind"] == "screen":
        z = net(X)
        r = torch.cat([torch.sigmoid(-z[:, :1]), torch.sigmoid(z[:, 1:])], 1)
        return r.reshape(case["designs"], case["jitter"], 2).mean(1)
    Y, flat = _labels(X32, seed).double(), [t for q in par for t in q]
    opt = torch.optim.AdamW([dict(params=flat[::2], weight_decay=TRAIN["weight_decay"]),
                             dict(params=flat[1::2], weight_decay=0.0)], lr=TRAIN["lr"], betas=(0.9, 0.999), eps=1e-8)
    for t in flat:
        t.requires_grad_(True)
    loss = []
    for lo in range(0, N, case["batch"]):
        opt.zero_grad()
        e = torch.nn.functional.binary_cross_entropy_with_logits(net(X[lo:lo + case["batch"]]), Y[lo:lo + case["batch"]])
        e.backward()
        opt.step()
        loss.append(e.detach())
    return dict(params=torch.cat([t.detach().reshape(-1) for t in flat]), loss=torch.stack(loss))


def _exact_kriging(case, seed):
    X, y, draws, far, near = _kriging(case, seed)
    n, d = X.shape
    Xt, yt = _t(X), _t(y)
    D2, one = (Xt[:, None] - Xt[None]) ** 2, torch.ones((n, 1), dtype=torch.float64, device=DEV)
    eye = 1e-10 * torch.eye(n, dtype=torch.float64, device=DEV)

    def fit(th):
        C, bad = torch.linalg.cholesky_ex(torch.exp(-(D2 @ th)) + eye)
        zw = torch.linalg.solve_triangular(C, torch.cat([yt[:, None], one], 1), upper=False)
        ww = (zw[:, 1] ** 2).sum()
        mu = (zw[:, 0] * zw[:, 1]).sum() / ww
        s2 = ((zw[:, 0] - mu * zw[:, 1]) ** 2).sum() / n
        v = n * torch.log(s2) + 2 * torch.log(torch.diagonal(C)).sum()
        return (math.inf if int(bad) else float(v)), C, mu, s2, ww

    best, best_v, lo, hi = None, math.inf, -3.0, 2.0
    for r, U in enumerate(draws):
        if r == 0:
            a, b = np.full(d, lo), np.full(d, hi)
        else:
            w = (hi - lo) / 2.0 ** (r + 1)
            a, b = np.maximum(best - w, lo), np.minimum(best + w, hi)
        cand = a + (b - a) * U
        v = [fit(_t(10.0 ** c))[0] for c in cand]
        j = int(np.argmin(v))
        if v[j] < best_v:
            best, best_v = cand[j], v[j]
    theta = 10.0 ** best
    _, C, mu, s2, ww = fit(_t(theta))
    b = X[int(np.argmin(y))]
    lo_, hi_ = np.clip(b - 0.05, 0.0, 1.0), np.clip(b + 0.05, 0.0, 1.0)
    pts = _t(np.concatenate([far, lo_ + (hi_ - lo_) * near]))
    r = torch.exp(-(((pts * _t(theta).sqrt())[:, None] - (Xt * _t(theta).sqrt())[None]) ** 2).sum(-1))
    solve = lambda rhs: torch.linalg.solve_triangular(C, rhs, upper=False)
    V, c, a = solve(r.T), solve(one), solve(yt[:, None] - mu)
    yhat = mu + (V * a).sum(0)
    s = (s2 * (1 - (V * V).sum(0) + (1 - (V * c).sum(0)) ** 2 / ww)).clamp(min=0).sqrt()
    f = float(y.min())
    z = (f - yhat) / s
    ei = (f - yhat) * 0.5 * (1 + torch.erf(z / math.sqrt(2))) + s * torch.exp(-0.5 * z * z) / math.sqrt(2 * math.pi)
    return dict(theta=theta, nll=best_v, yhat=yhat, s=s, ei=torch.where(s > 0, ei, (f - yhat).clamp(min=0)))
