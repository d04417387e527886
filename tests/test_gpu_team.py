"""Chains run by a team of warps (few chains: the line search's trial points are
evaluated at once) are bitwise the chains of the kernel that evaluates them one
after the other."""
import numpy as np
import pytest

from paper_2303_09916_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2303_09916_gb300 import dsdp  # noqa: E402

DEV, BOX, H = "cuda", 13.0, 0.375


class _Single:
    """One atom: no bonds, no pairs, no torsions."""

    def __init__(self, center):
        self.xyz = np.asarray(center, np.float32).reshape(1, 3)
        self.xs_type = np.array([0], np.uint8)
        self.bonds, self.rotatable = np.zeros((0, 2), np.int32), np.zeros(0, np.uint8)
        self.n_atoms, self.n_torsions = 1, 0


def _ligand(atoms, T, seed, center, kind):
    if atoms == 1:
        return _Single(center)
    lig = synth.ligand(atoms, T, seed, center=center)
    if kind == "carbon":  # every pair hydrophobic
        lig.xs_type[:] = synth.C_H
    if kind == "polar":  # no pair with a hydrophobic or H-bond term
        lig.xs_type[:] = synth.C_P
    return lig


# (atoms, torsions, pair kind, chains, MC steps, iterations, trace, site points, map type, map kind): teams of 8 for
# up to 152 chains in all, of 4 for up to 1,216; both lane layouts and their edges; one and two iterations
PLANS = [
    [(30, 8, "any", 3, 4, 100, 0, False, 0, 0)],
    [(1, 0, "any", 5, 2, 100, 1, False, 0, 0), (2, 0, "any", 1, 2, 100, 0, False, 0, 0), (9, 2, "polar", 9, 3, 40, 2, True, 0, 0),
     (32, 9, "carbon", 7, 2, 60, 1, False, 0, 0), (33, 9, "any", 7, 2, 60, 1, False, 0, 0), (64, 15, "polar", 3, 2, 30, 0, False, 0, 0)],
    [(20, 4, "any", 400, 2, 1, 1, False, 1, 0), (45, 11, "carbon", 300, 2, 2, 0, False, 2, 1), (30, 6, "any", 300, 2, 50, 1, True, 2, 1)],
]


def _jobs(spec, stream):
    rec = synth.receptor(1500, 12)
    xyz, ty = torch.from_numpy(rec.xyz).to(DEV), torch.from_numpy(rec.xs_type).to(DEV)
    box, n = dsdp.make_box(rec.pocket_center, BOX, H), [int(np.ceil(BOX / H))] * 3
    jobs, outs, keep, maps = [], [], [xyz, ty], {}
    for i, (atoms, T, kind, chains, steps, iters, trace, sites, dtype, mode) in enumerate(spec):
        if (dtype, mode) not in maps:
            nb = dsdp.dsdp_grid_map_bytes(box, dtype, mode)
            maps[dtype, mode] = torch.empty(nb, dtype=torch.uint8, device=DEV)
            dsdp.dsdp_grid_build_device(len(ty), xyz.data_ptr(), ty.data_ptr(), box, dtype, mode,
                                        maps[dtype, mode].data_ptr(), nb, stream)
        lig = _ligand(atoms, T, 30 + i, rec.pocket_center, kind)
        blob = dsdp.dsdp_ligand_pack(lig)
        nx = 7 + lig.n_torsions
        out = dict(conf=torch.zeros((chains, nx), device=DEV), e=torch.zeros(chains, device=DEV),
                   evals=torch.zeros(chains, dtype=torch.int32, device=DEV),
                   trace=torch.zeros((chains, steps + 1, nx + 4), device=DEV))
        p = dsdp.make_params(n_chains=chains, n_mc_steps=steps, n_opt_iters=iters, seed=70 + i, trace=trace,
                             site_points=synth.site_points(rec, 20, i) if sites else None)
        d_blob = torch.from_numpy(blob).to(DEV)
        j = dsdp.dsdp_job_device()
        j.grid = dsdp.grid_view(maps[dtype, mode].data_ptr(), n, [c - (n[0] - 1) * H / 2 for c in rec.pocket_center], H,
                                dtype, mode)
        j.h_blob, j.d_blob, j.params = blob.ctypes.data, d_blob.data_ptr(), p
        for a in range(3):
            j.box_lo[a], j.box_size[a] = rec.pocket_center[a] - BOX / 2, BOX
        if sites:
            pts = torch.from_numpy(p._keep_sites).to(DEV)
            j.d_site_points = pts.data_ptr()
            keep.append(pts)
        j.d_chain_best_conf, j.d_chain_best_e = out["conf"].data_ptr(), out["e"].data_ptr()
        j.d_chain_evals, j.d_trace = out["evals"].data_ptr(), out["trace"].data_ptr()
        jobs.append(j)
        outs.append(out)
        keep += [blob, d_blob, p]
    return jobs, outs, (keep, maps)


@pytest.mark.parametrize("spec", range(len(PLANS)))
def test_team_chains_are_the_single_warp_chains(spec):
    stream = torch.cuda.current_stream().cuda_stream
    jobs, outs, keep = _jobs(PLANS[spec], stream)
    got = []
    for tile_config in (1, 0, 0):  # 128 registers, one warp a chain; automatic, twice
        plan = dsdp.dsdp_plan_create(None, jobs, dsdp.DSDP_PLAN_NO_RESCORE, tile_config)
        dsdp.dsdp_plan_launch(plan, stream)
        torch.cuda.synchronize()
        got.append([{k: v.cpu().numpy().copy() for k, v in o.items()} for o in outs])
        for o in outs:
            for v in o.values():
                v.zero_()
        dsdp.dsdp_plan_destroy(None, plan)
    assert all(o["evals"].min() > 0 for o in got[0])
    for other in got[1:]:
        for i, (w, o) in enumerate(zip(got[0], other)):
            for k in w:
                assert np.array_equal(w[k], o[k], equal_nan=True), (i, k)
    # the autotuner leaves a plan that gives the same chains, whatever it keeps
    plan = dsdp.dsdp_plan_create(None, jobs, dsdp.DSDP_PLAN_NO_RESCORE, 0)
    chosen, ms = dsdp.dsdp_plan_autotune(plan, stream, 1, with_times=True)
    assert 1 <= chosen <= 24 and chosen in ms
    dsdp.dsdp_plan_launch(plan, stream)
    torch.cuda.synchronize()
    for w, o in zip(got[0], outs):
        assert all(np.array_equal(w[k], o[k].cpu().numpy(), equal_nan=True) for k in w)
    dsdp.dsdp_plan_destroy(None, plan)
