"""Timed cases of the docking path: the calls a program that docks ligands makes,
through the public entry points, from a handful of poses to a screening batch.

Every case is a dict of plain values whose "kind" names the entry point:

  score    dsdp_score_eval_device: score + gradient of a batch of conformations
  grid     dsdp_grid_build_device: the score (+ gradient) maps of one receptor
  voxel    dsdp_voxelize_device: the receptor's voxel features
  rescore  dsdp_plan_launch_stage(RESCORE): FP64 rescoring + top-k of given poses
  dock     dsdp_plan_launch: chains, FP64 rescoring and top-k of one batch of jobs
  host     dsdp_dock_submit_many + dsdp_dock_poll: the same through host arrays

Receptors and ligands come from the package's seeded generators.  The maps that
the score, dock and host cases read are inputs like them: plain torch makes them
here, in FP32 (a program keeps the maps of the receptor it screens against, and
a Monte Carlo search amplifies any difference in them), rounded to the case's
map type.  `exact` restates each computation in FP64.
"""
import math

import numpy as np
import torch

from paper_2303_09916_gb300 import dsdp, synth

DEV = "cuda"
DTYPES = {"f32": (dsdp.DSDP_MAP_F32, torch.float32), "bf16": (dsdp.DSDP_MAP_BF16, torch.bfloat16),
          "f16": (dsdp.DSDP_MAP_F16, torch.float16)}
MODES = {"eq4": dsdp.DSDP_GRID_EQ4, "eq3": dsdp.DSDP_GRID_EQ3}
TOP_K = 9


# ------------------------------------------------------------------ the cases
def _dock(name, **kw):
    c = dict(name=name, kind="dock", n_rec=4000, box=30.0, jobs=1, atoms_lo=30, atoms_hi=30, tors_lo=8, tors_hi=8,
             chains=384, steps=40, opt="bfgs", map="f32", mode="eq4", sites=False)
    c.update(kw)
    return c


def listed():
    return [
        # a few poses looked at in an interactive session or a minimiser's step: launch and latency
        dict(name="score_poses_32", kind="score", n_conf=32, atoms=30, torsions=8, n_rec=4000, box=30.0, map="f32",
             mode="eq4"),
        # re-scoring a pose library of drug-like to large ligands on the serving map format
        dict(name="score_library_100k", kind="score", n_conf=100003, atoms=45, torsions=11, n_rec=4000, box=30.0,
             map="bf16", mode="eq4"),
        # maps of a small receptor around a known site (54^3, odd against the kernel's bricks)
        dict(name="grid_2k_f32", kind="grid", n_rec=2000, box=20.0, map="f32", mode="eq4"),
        # the largest serving receptor and box (107^3), 16-bit maps
        dict(name="grid_8k_bf16", kind="grid", n_rec=8000, box=40.0, map="bf16", mode="eq4"),
        # binding-site network input of a typical receptor
        dict(name="voxel_4k", kind="voxel", n_rec=4000),
        # postprocess of a batch: best poses of 8 jobs scored exactly and ranked
        dict(name="rescore_8x384", kind="rescore", n_rec=4000, jobs=8, chains=384, atoms=30, torsions=8),
        # the small workload: one system, 64 chains x 100 steps in a 20 A box (latency of one request)
        _dock("dock_plain_2k", n_rec=2000, box=20.0, atoms_lo=20, atoms_hi=20, tors_lo=4, tors_hi=4, chains=64,
              steps=100),
        # the typical system alone: one request on an idle GPU
        _dock("dock_typical_4k"),
        # screening: 16 ligands against one receptor in one launch, the GPU full
        _dock("dock_screen_16", jobs=16),
        # uneven library on 16-bit maps: 10-60 atoms, 0-15 torsions, 128 chains each
        _dock("dock_uneven_64", n_rec=5000, box=26.0, jobs=64, atoms_lo=10, atoms_hi=60, tors_lo=0, tors_hi=15,
              chains=128, map="bf16"),
        # Barzilai-Borwein (the paper's optimiser) in the adaptive search space, FP16 maps
        _dock("dock_bb_sites", jobs=4, chains=512, steps=20, opt="bb", map="f16", sites=True),
        # the whole call from host arrays: submit six ligands together, fetch every result
        dict(name="host_screen_6", kind="host", n_rec=4000, box=30.0, jobs=6, atoms_lo=20, atoms_hi=36, tors_lo=4,
             tors_hi=10, chains=256, steps=20, opt="bfgs", map="f32", mode="eq4", sites=False),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["score", "score", "grid", "grid", "voxel", "rescore", "dock", "dock", "dock", "host"])
    fmt = dict(map=rng.choice(["f32", "bf16", "f16"]), mode=rng.choice(["eq4", "eq4", "eq3"]))
    n_rec = _log(rng, 500, 8000)
    box = round(rng.uniform(12.0, 36.0), 2)
    if kind == "score":
        atoms = rng.randint(6, 64)
        return dict(kind=kind, n_conf=_log(rng, 1, 100000), atoms=atoms,
                    torsions=rng.randint(0, min(15, max(0, atoms // 2 - 2))), n_rec=n_rec, box=box, **fmt)
    if kind == "grid":
        return dict(kind=kind, n_rec=n_rec, box=box, **fmt)
    if kind == "voxel":
        return dict(kind=kind, n_rec=n_rec)
    if kind == "rescore":
        atoms, jobs = rng.randint(8, 60), _log(rng, 1, 12)
        return dict(kind=kind, n_rec=_log(rng, 500, 6000), jobs=jobs, chains=_log(rng, 16, 3072 // jobs), atoms=atoms,
                    torsions=rng.randint(0, min(15, max(0, atoms // 2 - 2))))
    lo = rng.randint(8, 50)
    hi = rng.randint(lo, 60)
    c = dict(kind=kind, n_rec=n_rec, box=box, jobs=_log(rng, 1, 6 if kind == "host" else 24), atoms_lo=lo, atoms_hi=hi,
             tors_lo=rng.randint(0, 4), tors_hi=rng.randint(4, 15), steps=_log(rng, 4, 60),
             opt=rng.choice(["bfgs", "bfgs", "bb"]), sites=rng.random() < 0.3, **fmt)
    # at most half the largest listed case's chains x steps x pairs
    most = int(1.2e8 / (c["jobs"] * c["steps"] * hi * hi * (2 if c["opt"] == "bb" else 1)))
    c["chains"] = _log(rng, 8, max(16, min(1024, most)))
    return c


# ------------------------------------------------------------------ inputs
class _State:
    """Inputs and handles of one case; the handles go with it."""

    def __init__(self, case):
        self.case = case
        self.ctx = self.plan = self.grid = None

    def __del__(self):
        if self.plan:
            torch.cuda.synchronize()
            dsdp.dsdp_plan_destroy(None, self.plan)
        if self.ctx:
            dsdp.dsdp_grid_free(self.ctx, self.grid)
            dsdp.dsdp_destroy(self.ctx)


def _seed(seed):
    return int(seed) % 1000003


def _receptor(case, seed):
    return synth.receptor(case["n_rec"], _seed(seed))


def _box(rec, case):
    return dsdp.make_box(rec.pocket_center, case["box"], 0.375)


def _geometry(rec, case):
    n = int(math.ceil(case["box"] / 0.375))
    return n, np.array([rec.pocket_center[a] - (n - 1) * 0.375 / 2.0 for a in range(3)])


def _ligands(case, seed, center):
    """One ligand per job; the sizes belong to the case, trees and types to the seed.  A tree of n atoms with at
    most three bonds each has at least n / 2 - 2 bonds that can rotate."""
    rng = np.random.default_rng([case["jobs"], case["atoms_lo"], case["atoms_hi"]])
    out = []
    for i in range(case["jobs"]):
        n = int(rng.integers(case["atoms_lo"], case["atoms_hi"] + 1))
        t = int(rng.integers(case["tors_lo"], case["tors_hi"] + 1))
        out.append(synth.ligand(n, min(t, max(0, n // 2 - 2)), _seed(seed) * 64 + i, center=center))
    return out


def _confs(rec, lig, n, seed, spread=2.0):
    """n poses around the pocket: position, unit quaternion, torsions in (-pi, pi]; FP32."""
    rng = np.random.default_rng([_seed(seed), 9])
    T = lig.n_torsions
    c = np.empty((n, 7 + T))
    c[:, :3] = rec.pocket_center + rng.uniform(-spread, spread, (n, 3))
    q = rng.normal(size=(n, 4))
    c[:, 3:7] = q / np.linalg.norm(q, axis=1, keepdims=True)
    c[:, 7:] = rng.uniform(-math.pi, math.pi, (n, T))
    return c.astype(np.float32)


RADIUS = [1.9, 1.9, 1.8, 1.8, 1.8, 1.7, 1.7, 2.0, 1.8]
HYD = [1, 0, 0, 0, 0, 0, 0, 0, 0]
DON = [0, 0, 0, 1, 0, 0, 1, 0, 1]
ACC = [0, 0, 0, 0, 1, 1, 1, 0, 1]


def _pair(d, hyd, hb):
    """Vina pair terms of surface distance d and their slopes; hyd / hb: 0-1 weights that broadcast."""
    g1, g2 = torch.exp(-4.0 * d * d), torch.exp(-0.25 * (d - 3.0) ** 2)
    m = d.clamp(max=0.0)
    e = -0.0356 * g1 - 0.00516 * g2 + 0.840 * m * m
    s = 0.0356 * 8.0 * d * g1 + 0.00516 * 0.5 * (d - 3.0) * g2 + 1.680 * m
    if hyd is not None:
        e = e - 0.0351 * hyd * (1.5 - d).clamp(0.0, 1.0)
        s = s + 0.0351 * hyd * ((d >= 0.5) & (d < 1.5))
    if hb is not None:
        e = e - 0.587 * hb * (d / -0.7).clamp(0.0, 1.0)
        s = s + (0.587 / 0.7) * hb * ((d >= -0.7) & (d < 0.0))
    return e, s


def _maps(rec, case, dtype):
    """The eight maps [type][z][y][x][channel] of a receptor in plain torch, block by block of vertex rows."""
    n, origin = _geometry(rec, case)
    ch = 4 if case["mode"] == "eq4" else 1
    out = torch.empty((8, n, n, n, ch), dtype=dtype, device=DEV)
    ax = [torch.tensor(origin[a] + 0.375 * np.arange(n), dtype=dtype, device=DEV) for a in range(3)]
    xyz_h, ty_h = rec.xyz.astype(np.float64), rec.xs_type.astype(np.int64)
    by, bz = 8, 16
    for z0 in range(0, n, bz):
        for y0 in range(0, n, by):
            z1, y1 = min(z0 + bz, n), min(y0 + by, n)
            lo = np.array([origin[0], origin[1] + 0.375 * y0, origin[2] + 0.375 * z0])
            hi = np.array([origin[0] + 0.375 * (n - 1), origin[1] + 0.375 * (y1 - 1), origin[2] + 0.375 * (z1 - 1)])
            gap = np.maximum(np.maximum(lo - xyz_h, xyz_h - hi), 0.0)
            near = np.nonzero((gap * gap).sum(1) < 8.01 ** 2)[0]
            view = out[:, z0:z1, y0:y1]
            if not len(near):
                view.zero_()
                continue
            p = torch.from_numpy(xyz_h[near]).to(DEV).to(dtype)
            t = ty_h[near]
            rj = torch.tensor([RADIUS[k] for k in t], dtype=dtype, device=DEV)
            fl = lambda table: torch.tensor([float(table[k]) for k in t], dtype=dtype, device=DEV)  # noqa: E731
            hyd, don, acc = fl(HYD), fl(DON), fl(ACC)
            gz, gy, gx = torch.meshgrid(ax[2][z0:z1], ax[1][y0:y1], ax[0], indexing="ij")
            dx, dy, dz = ((g.reshape(-1, 1) - p[None, :, a]) for a, g in enumerate((gx, gy, gz)))
            r2 = dx * dx + dy * dy + dz * dz
            r = torch.sqrt(r2)
            inside = r2 < 64.0
            inv = torch.where(r > 0, 1.0 / r, torch.zeros_like(r))
            u = [dx * inv, dy * inv, dz * inv] if ch == 4 else []
            del dx, dy, dz, r2, inv
            for radius, members in ((1.9, (0, 1)), (1.8, (2, 3, 4)), (1.7, (5, 6)), (2.0, (7,))):
                d = torch.where(inside, r - (radius + rj), torch.full_like(r, 100.0))
                for k in members:
                    h = hyd if HYD[k] else None
                    b = (acc if DON[k] and not ACC[k] else don if ACC[k] and not DON[k] else torch.maximum(don, acc)) \
                        if DON[k] or ACC[k] else None
                    e, s = _pair(d, h, b)
                    cols = [e.sum(1)] + [(s * w).sum(1) for w in u]
                    view[k] = torch.stack(cols, -1).reshape(z1 - z0, y1 - y0, n, ch)
    return out


class _MapSet:
    """A receptor on the device with its maps in the case's format."""

    def __init__(self, case, seed):
        self.rec = _receptor(case, seed)
        self.n, self.origin = _geometry(self.rec, case)
        self.code, tdtype = DTYPES[case["map"]]
        self.mode = MODES[case["mode"]]
        self.maps = _maps(self.rec, case, torch.float32).to(tdtype)
        self.xyz = torch.from_numpy(self.rec.xyz).to(DEV)
        self.type = torch.from_numpy(self.rec.xs_type).to(DEV)

    def view(self):
        return dsdp.grid_view(self.maps.data_ptr(), [self.n] * 3, self.origin, 0.375, self.code, self.mode)


def _params(case, seed, i, rec):
    sites = synth.site_points(rec, 100, _seed(seed)) if case.get("sites") else None
    return dsdp.make_params(n_chains=case["chains"], n_mc_steps=case.get("steps", 1), seed=int(seed) * 7919 + i,
                            optimizer=dsdp.DSDP_OPT_BB if case.get("opt") == "bb" else dsdp.DSDP_OPT_BFGS,
                            top_k=TOP_K, site_points=sites)


def _plan(s, case, seed, m, ligs, confs=None):
    """Jobs of one batch with caller-owned outputs, and their plan; confs: given poses per job (rescoring)."""
    s.m, s.keep, jobs, J, C = m, [], [], len(ligs), case["chains"]
    n_at = [x.n_atoms for x in ligs]
    nx = [7 + x.n_torsions for x in ligs]
    z = lambda shape, dt: torch.zeros(shape, dtype=dt, device=DEV)  # noqa: E731
    s.n, s.chain = z(J, torch.int32), z((J, TOP_K), torch.int32)
    s.score, s.inter, s.intra = (z((J, TOP_K), torch.float64) for _ in range(3))
    s.conf, s.coords = z(TOP_K * sum(nx), torch.float64), z(TOP_K * sum(n_at) * 3, torch.float32)
    s.best_e, s.evals, s.best = z((J, C), torch.float32), z((J, C), torch.int32), z(C * sum(nx), torch.float32)
    size = float(case.get("box", 20.0))
    at = lambda t, k: t.data_ptr() + k * t.element_size()  # noqa: E731
    o_nx = o_at = 0
    for i, lig in enumerate(ligs):
        blob = dsdp.dsdp_ligand_pack(lig)
        d_blob = torch.from_numpy(blob).to(DEV)
        p = _params(case, seed, i, m.rec)
        j = dsdp.dsdp_job_device()
        j.grid = m.view()
        j.receptor = dsdp.dsdp_receptor(len(m.rec.xs_type), m.xyz.data_ptr(), m.type.data_ptr())
        j.h_blob, j.d_blob, j.params = blob.ctypes.data, d_blob.data_ptr(), p
        for a in range(3):
            j.box_lo[a], j.box_size[a] = m.rec.pocket_center[a] - size / 2, size
        s.keep += [blob, d_blob, p]
        if p.n_site_points:
            pts = torch.from_numpy(p._keep_sites).to(DEV)
            j.d_site_points = pts.data_ptr()
            s.keep.append(pts)
        if confs is not None:
            s.best[C * o_nx: C * (o_nx + nx[i])] = torch.from_numpy(confs[i]).to(DEV).reshape(-1)
        j.d_chain_best_conf, j.d_chain_best_e = at(s.best, C * o_nx), at(s.best_e, i * C)
        j.d_chain_evals, j.d_out_n = at(s.evals, i * C), at(s.n, i)
        j.d_out_chain, j.d_out_score = at(s.chain, i * TOP_K), at(s.score, i * TOP_K)
        j.d_out_inter, j.d_out_intra = at(s.inter, i * TOP_K), at(s.intra, i * TOP_K)
        j.d_out_conf, j.d_out_coords = at(s.conf, TOP_K * o_nx), at(s.coords, TOP_K * 3 * o_at)
        o_nx, o_at = o_nx + nx[i], o_at + n_at[i]
        jobs.append(j)
    s.plan = dsdp.dsdp_plan_create(None, jobs, 0, 0)


def prepare(case, seed):
    s = _State(case)
    kind = case["kind"]
    if kind == "score":
        s.m = _MapSet(case, seed)
        s.lig = synth.ligand(case["atoms"], case["torsions"], _seed(seed), center=s.m.rec.pocket_center)
        s.blob = dsdp.dsdp_ligand_pack(s.lig)
        s.d_blob = torch.from_numpy(s.blob).to(DEV)
        s.confs = torch.from_numpy(_confs(s.m.rec, s.lig, case["n_conf"], seed)).to(DEV)
        s.e = torch.empty(case["n_conf"], device=DEV)
        s.g = torch.empty((case["n_conf"], 6 + s.lig.n_torsions), device=DEV)
        s.view = s.m.view()
    elif kind == "grid":
        rec = _receptor(case, seed)
        n, _ = _geometry(rec, case)
        code, tdtype = DTYPES[case["map"]]
        s.box, s.code, s.mode = _box(rec, case), code, MODES[case["mode"]]
        s.xyz, s.type = torch.from_numpy(rec.xyz).to(DEV), torch.from_numpy(rec.xs_type).to(DEV)
        s.maps = torch.empty((8, n, n, n, 4 if case["mode"] == "eq4" else 1), dtype=tdtype, device=DEV)
    elif kind == "voxel":
        rec = _receptor(case, seed)
        s.center = synth.protein_center(rec)
        s.inputs = [torch.from_numpy(np.ascontiguousarray(a)).to(DEV)
                    for a in (rec.xyz, *synth.receptor_voxel_inputs(rec))]
        s.work = torch.empty(dsdp.dsdp_voxel_work_bytes(), dtype=torch.uint8, device=DEV)
        s.out = torch.empty((36, 36, 36, 18), device=DEV)
    elif kind == "rescore":
        m = _State(case)
        m.rec = _receptor(case, seed)
        m.xyz, m.type = torch.from_numpy(m.rec.xyz).to(DEV), torch.from_numpy(m.rec.xs_type).to(DEV)
        m.node = torch.zeros(8 * 8 * 4, device=DEV)  # rescoring is gridless: the smallest grid stands in
        m.view = lambda: dsdp.grid_view(m.node.data_ptr(), [2] * 3, m.rec.pocket_center, 0.375)
        s.ligs, s.poses = _rescore_inputs(case, seed, m.rec)
        _plan(s, case, seed, m, s.ligs, s.poses)
    elif kind == "dock":
        m = _MapSet(case, seed)
        _plan(s, case, seed, m, _ligands(case, seed, m.rec.pocket_center))
    elif kind == "host":
        m = _MapSet(case, seed)
        s.ligs = _ligands(case, seed, m.rec.pocket_center)
        s.params = [_params(case, seed, i, m.rec) for i in range(case["jobs"])]
        s.ctx = dsdp.dsdp_create(0)
        s.grid = dsdp.dsdp_grid_from_maps(s.ctx, m.rec.xyz, m.rec.xs_type, _box(m.rec, case), m.code, m.mode,
                                          m.maps.float().cpu().numpy())
    else:
        raise ValueError(kind)
    return s


def _rescore_inputs(case, seed, rec):
    ligs = [synth.ligand(case["atoms"], case["torsions"], _seed(seed) * 64 + i, center=rec.pocket_center)
            for i in range(case["jobs"])]
    return ligs, [_confs(rec, x, case["chains"], seed * 64 + i) for i, x in enumerate(ligs)]


# ------------------------------------------------------------------ one pass
def run(s):
    kind = s.case["kind"]
    st = torch.cuda.current_stream().cuda_stream
    if kind == "score":
        dsdp.dsdp_score_eval_device(s.view, s.blob, s.d_blob.data_ptr(), s.confs.data_ptr(), s.case["n_conf"],
                                    s.e.data_ptr(), s.g.data_ptr(), dsdp.DSDP_TERM_ALL, st)
        return {"energy": s.e, "grad": s.g}
    if kind == "grid":
        dsdp.dsdp_grid_build_device(s.type.numel(), s.xyz.data_ptr(), s.type.data_ptr(), s.box, s.code, s.mode,
                                    s.maps.data_ptr(), s.maps.numel() * s.maps.element_size(), st)
        return {"maps": s.maps}
    if kind == "voxel":
        x, r, f = s.inputs
        dsdp.dsdp_voxelize_device(len(r), x.data_ptr(), r.data_ptr(), f.data_ptr(), s.center, s.out.data_ptr(),
                                  s.work.data_ptr(), s.work.numel(), st)
        return {"voxels": s.out}
    if kind == "host":
        c = s.case
        ids = dsdp.dsdp_dock_submit_many(s.ctx, [s.grid] * c["jobs"], s.ligs, s.params)
        out = []
        for i, lig, p in zip(ids, s.ligs, s.params):
            bufs = dsdp.result_buffers(lig.n_atoms, lig.n_torsions, p)
            r = dsdp.dsdp_dock_poll(s.ctx, i, bufs)
            out.append({**bufs, "n_out": r["n_out"], "n_evals": r["n_evals"]})
        return out
    top = {"n": s.n, "chain": s.chain, "score": s.score, "inter": s.inter, "intra": s.intra, "conf": s.conf,
           "coords": s.coords}
    if kind == "rescore":
        dsdp.dsdp_plan_launch_stage(s.plan, dsdp.DSDP_STAGE_RESCORE, st)
        return top
    dsdp.dsdp_plan_launch(s.plan, st)
    return {**top, "best_e": s.best_e, "best_conf": s.best, "evals": s.evals}


# ------------------------------------------------------------------ necessary work
def work(case):
    kind = case["kind"]
    if kind == "voxel":
        # features and positions in, voxels out; per atom 98 points against the about 60 spheres that reach them
        return {"bytes": 4 * (21 * case["n_rec"] + 36 ** 3 * 18), "flops": case["n_rec"] * 98 * 60 * 8}
    if kind == "rescore":
        pairs = case["atoms"] * 85  # receptor atoms within 8 A of a ligand atom in the pocket (protein: 107)
        n = case["jobs"] * case["chains"]
        return {"bytes": 13 * case["n_rec"] + n * 4 * (7 + case["torsions"]), "flops": n * pairs * 60}
    n = math.ceil(case["box"] / 0.375)
    node = (4 if case["mode"] == "eq4" else 1) * (4 if case["map"] == "f32" else 2)
    if kind == "grid":
        # each vertex: about 85 receptor atoms within 8 A, four radii, two exponentials and the gradient each
        return {"bytes": 8 * n ** 3 * node + 13 * case["n_rec"], "flops": n ** 3 * 85 * 4 * 30}
    if kind == "score":
        evals, sizes = case["n_conf"], [case["atoms"]]
        io = evals * 4 * (7 + case["torsions"] + 7 + case["torsions"])
    else:
        # evaluations of a local optimisation: 62 on average with BFGS, 101 with Barzilai-Borwein
        per = 62 if case["opt"] == "bfgs" else 101
        evals = case["jobs"] * case["chains"] * (case["steps"] + 1) * per
        k = case["jobs"]
        sizes = [case["atoms_lo"] + (case["atoms_hi"] - case["atoms_lo"]) * (i + 0.5) / k for i in range(k)]
        io = case["jobs"] * case["chains"] * 4 * 20
    # three quarters of an atom pair list are intra pairs; 40 flop a pair, 120 an atom
    flops = evals * sum(40 * 0.75 * a * (a - 1) / 2 + 120 * a for a in sizes) / len(sizes)
    gathers = evals * sum(sizes) / len(sizes) * 8 * node
    return {"bytes": io + min(8 * n ** 3 * node, gathers), "flops": flops}


# ------------------------------------------------------------------ FP64 restatement
class _Tree:
    """Rigid bodies and torsion tree of a ligand, and its atom positions for a batch of conformations."""

    def __init__(self, lig):
        n = lig.n_atoms
        rot = [tuple(b) for b, f in zip(lig.bonds.tolist(), lig.rotatable) if f]
        rigid = [[] for _ in range(n)]
        full = [[] for _ in range(n)]
        for (i, j), f in zip(lig.bonds.tolist(), lig.rotatable):
            full[i].append(j), full[j].append(i)
            if not f:
                rigid[i].append(j), rigid[j].append(i)
        self.body = self._components(n, rigid)
        sizes = [self.body.count(b) for b in range(max(self.body) + 1)]
        root = sizes.index(max(sizes))
        self.order, self.n = [(root, None, None, self.body.index(root), None)], n
        for b, *_ in self.order:  # grows while it is walked
            for k, (i, j) in enumerate(rot):
                near, far = (i, j) if self.body[i] == b else (j, i)
                if self.body[near] == b and self.body[far] not in [o[0] for o in self.order]:
                    self.order.append((self.body[far], b, k, far, near))
        dist = [self._distances(n, full, i) for i in range(n)]
        self.pairs = [(i, j) for i in range(n) for j in range(i + 1, n)
                      if self.body[i] != self.body[j] and dist[i][j] > 3]
        self.ref = torch.tensor(lig.xyz.astype(np.float64), device=DEV)
        self.T, self.type = len(rot), lig.xs_type.tolist()

    @staticmethod
    def _components(n, adj):
        comp, c = [-1] * n, 0
        for s in range(n):
            if comp[s] < 0:
                todo, comp[s] = [s], c
                while todo:
                    for y in adj[todo.pop()]:
                        if comp[y] < 0:
                            comp[y] = c
                            todo.append(y)
                c += 1
        return comp

    @staticmethod
    def _distances(n, adj, s):
        d, todo = [n] * n, [s]
        d[s] = 0
        for x in todo:
            for y in adj[x]:
                if d[y] == n:
                    d[y] = d[x] + 1
                    todo.append(y)
        return d

    def positions(self, conf, theta):
        q = conf[:, 3:7] / conf[:, 3:7].norm(dim=1, keepdim=True)
        w, x, y, z = q.unbind(1)
        R = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                         2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                         2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], 1).reshape(-1, 3, 3)
        frames, out = {}, [None] * self.n
        for b, parent, k, origin, near in self.order:
            if parent is None:
                rot, at = R, conf[:, :3]
            else:
                rp, op, o0 = frames[parent]
                a = self.ref[origin] - self.ref[near]
                a = a / a.norm()
                K = torch.tensor([[0, -a[2], a[1]], [a[2], 0, -a[0]], [-a[1], a[0], 0]], dtype=a.dtype, device=DEV)
                t = theta[:, k, None, None]
                rot = rp @ (torch.eye(3, dtype=a.dtype, device=DEV) + torch.sin(t) * K + (1 - torch.cos(t)) * (K @ K))
                at = op + (rp @ (self.ref[origin] - o0))
            frames[b] = (rot, at, self.ref[origin])
            for i in range(self.n):
                if self.body[i] == b:
                    out[i] = at + rot @ (self.ref[i] - self.ref[origin])
        return torch.stack(out, 1)

    def intra(self, pos, grad=False):
        """Pair energies [conf] and, with grad, atom gradients."""
        if not self.pairs:
            return pos.new_zeros(len(pos)), torch.zeros_like(pos)
        ij = torch.tensor(self.pairs, device=DEV).T
        ti, tj = ([self.type[k] for k in side] for side in ij.tolist())
        f = lambda v: torch.tensor([float(x) for x in v], dtype=pos.dtype, device=DEV)  # noqa: E731
        rr = f([RADIUS[a] + RADIUS[b] for a, b in zip(ti, tj)])
        hyd = f([HYD[a] and HYD[b] for a, b in zip(ti, tj)])
        hb = f([bool((DON[a] and ACC[b]) or (ACC[a] and DON[b])) for a, b in zip(ti, tj)])
        v = pos[:, ij[0]] - pos[:, ij[1]]
        r = v.norm(dim=2)
        e, sl = _pair(torch.where(r < 8.0, r - rr, torch.full_like(r, 100.0)), hyd, hb)
        g = torch.zeros_like(pos)
        if grad:
            w = (sl / r)[..., None] * v
            g.index_add_(1, ij[0], w).index_add_(1, ij[1], -w)
        return e.sum(1), g


def _inter_grid(m, case, tree, pos):
    """Trilinear score and gradient (Eq. 2 with Eq. 4 or Eq. 3) with the wall outside the grid."""
    origin = torch.tensor(m.origin, dtype=pos.dtype, device=DEV)
    u = (pos - origin) / 0.375
    c = u.clamp(0.0, float(m.n - 1))
    cell = c.floor().clamp(max=m.n - 2).long()
    f = c - cell
    ty = torch.tensor(tree.type, device=DEV)
    e, g = pos.new_zeros(pos.shape[:2]), torch.zeros_like(pos)
    for bits in range(8):
        b = [bits & 1, bits >> 1 & 1, bits >> 2 & 1]
        v = m.maps[ty, cell[..., 2] + b[2], cell[..., 1] + b[1], cell[..., 0] + b[0]].to(pos.dtype)
        w = [f[..., a] if b[a] else 1 - f[..., a] for a in range(3)]
        e += w[0] * w[1] * w[2] * v[..., 0]
        if case["mode"] == "eq4":
            g += (w[0] * w[1] * w[2])[..., None] * v[..., 1:]
        else:
            for a in range(3):
                o = [k for k in range(3) if k != a]
                g[..., a] += (1 if b[a] else -1) / 0.375 * w[o[0]] * w[o[1]] * v[..., 0]
    ex = (u - c) * 0.375
    e = e + 10.0 * ex.abs().sum(2)
    return e.sum(1), torch.where(ex != 0, 10.0 * ex.sign(), g)


def _exact_score(case, seed):
    m = _MapSet(case, seed)
    lig = synth.ligand(case["atoms"], case["torsions"], _seed(seed), center=m.rec.pocket_center)
    tree = _Tree(lig)
    confs = torch.from_numpy(_confs(m.rec, lig, case["n_conf"], seed)).to(DEV).double()
    es, gs = [], []
    for c in confs.split(8192):
        th = c[:, 7:].clone().requires_grad_(True)
        pos = tree.positions(c, th)
        x = pos.detach()
        e1, g1 = _inter_grid(m, case, tree, x)
        e2, g2 = tree.intra(x, grad=True)
        g = g1 + g2
        parts = [g.sum(1), torch.linalg.cross(x - c[:, None, :3], g).sum(1)]
        if tree.T:
            parts.append(torch.autograd.grad((pos * g).sum(), th)[0])
        es.append(e1 + e2)
        gs.append(torch.cat(parts, 1))
    return {"energy": torch.cat(es), "grad": torch.cat(gs)}


def _exact_rescore(case, seed):
    rec = _receptor(case, seed)
    ligs, poses = _rescore_inputs(case, seed, rec)
    xyz = torch.from_numpy(rec.xyz).to(DEV).double()
    f = lambda v: torch.tensor([float(x) for x in v], dtype=torch.float64, device=DEV)  # noqa: E731
    rt = rec.xs_type.tolist()
    out = {k: [] for k in ("n", "chain", "score", "inter", "intra", "conf", "coords")}
    for lig, pose in zip(ligs, poses):
        tree = _Tree(lig)
        c = torch.from_numpy(pose).to(DEV).double()
        pos = tree.positions(c, c[:, 7:])
        intra, _ = tree.intra(pos)
        inter = torch.zeros_like(intra)
        for i, t in enumerate(tree.type):
            r = torch.cdist(pos[:, i], xyz, compute_mode="donot_use_mm_for_euclid_dist")
            rr = f([RADIUS[t] + RADIUS[k] for k in rt])
            hyd = f([HYD[t] and HYD[k] for k in rt])
            hb = f([bool((DON[t] and ACC[k]) or (ACC[t] and DON[k])) for k in rt])
            inter += _pair(torch.where(r < 8.0, r - rr, torch.full_like(r, 100.0)), hyd, hb)[0].sum(1)
        score = inter / (1.0 + 0.0585 * tree.T)
        kept = []
        for k in torch.sort(score, stable=True)[1].tolist():
            if len(kept) == TOP_K:
                break
            if all(float(((pos[k] - pos[o]) ** 2).sum()) >= tree.n for o in kept):
                kept.append(k)
        pad = lambda v: torch.cat([v, v.new_zeros((TOP_K - len(kept), *v.shape[1:]))])  # noqa: E731
        at = torch.tensor(kept, device=DEV)
        out["n"].append(torch.tensor(len(kept), dtype=torch.int32, device=DEV))
        out["chain"].append(pad(at.int()))
        for name, v in (("score", score), ("inter", inter), ("intra", intra)):
            out[name].append(pad(v[at]))
        out["conf"].append(pad(c[at]).reshape(-1))
        out["coords"].append(pad(pos[at]).reshape(-1))
    return {k: torch.cat(v) if k in ("conf", "coords") else torch.stack(v) for k, v in out.items()}


def _exact_voxel(case, seed):
    rec = _receptor(case, seed)
    n = case["n_rec"]
    radius, feats = synth.receptor_voxel_inputs(rec)
    lo = torch.tensor([float(np.float32(v - 35.0)) for v in synth.protein_center(rec)], device=DEV)
    xyz = torch.from_numpy(rec.xyz).to(DEV)
    cell = ((xyz - lo) * torch.tensor(np.float32(36.0) / np.float32(70.0), device=DEV)).floor().long()
    dirs = np.array([(a, b, c) for a in range(-2, 3) for b in range(-2, 3) for c in range(-2, 3)
                     if math.gcd(math.gcd(abs(a), abs(b)), abs(c)) == 1], dtype=np.float32)
    u = torch.from_numpy(dirs / np.sqrt((dirs * dirs).sum(1, dtype=np.float32))[:, None]).to(DEV)
    R = torch.from_numpy(radius).to(DEV) + 1.4
    surface = torch.zeros(n, dtype=torch.float64, device=DEV)
    for i0 in range(0, n, 128):
        i = torch.arange(i0, min(i0 + 128, n), device=DEV)
        p = xyz[i, None] + R[i, None, None] * u[None]
        d = [p[..., a, None] - xyz[None, None, :, a] for a in range(3)]
        hit = (d[0] * d[0] + d[1] * d[1]) + d[2] * d[2] < R * R
        hit[torch.arange(len(i), device=DEV), :, i] = False
        surface[i] = (~hit.any(2)).any(1).double()
    rows = torch.cat([torch.from_numpy(feats).to(DEV).double(), surface[:, None]], 1)
    ok = ((cell >= 0) & (cell < 36)).all(1)
    out = torch.zeros((36 ** 3, 18), dtype=torch.float64, device=DEV)
    out.index_add_(0, (cell[ok, 2] * 36 + cell[ok, 1]) * 36 + cell[ok, 0], rows[ok])
    return {"voxels": out.reshape(36, 36, 36, 18)}


def exact(case, seed):
    kind = case["kind"]
    if kind == "grid":
        return {"maps": _maps(_receptor(case, seed), case, torch.float64)}
    if kind == "score":
        return _exact_score(case, seed)
    if kind == "rescore":
        return _exact_rescore(case, seed)
    if kind == "voxel":
        return _exact_voxel(case, seed)
    return None  # a Monte Carlo search separates from any restatement of it at the first rounding
