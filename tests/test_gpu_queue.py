"""The time-sliced work queue of the chain stage (more chains than fit on the GPU at
once): chains run in slices, handed from CTA to CTA, in several launches that
overlap; the results are bitwise those of the launch that runs each chain to its
end."""
import numpy as np
import pytest

from paper_2303_09916_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2303_09916_gb300 import dsdp  # noqa: E402

BOX, H = 14.0, 0.375
# (atoms, torsions, map format, chains, MC steps, optimiser): more than 20 x 152 chains in each group of the first two;
# chain counts that leave part-filled tiles, ligands of less than 10 atoms (their records outgrow the coordinates),
# one MC step (a single-slice chain beside many-slice ones).  The first set outnumbers the chains' places; the others
# have a place for each, and their slowest chains are finished by teams of warps: of one tile size with
# Barzilai-Borwein chains among them, and of both
FEW = [[(30, 8, 0, 900, 5, 0), (24, 5, 0, 600, 3, 0), (32, 6, 0, 300, 4, 1)],
       [(20, 4, 1, 700, 6, 0), (60, 15, 1, 500, 3, 0), (33, 8, 1, 300, 2, 0)]]
JOBS = [(30, 8, 0, 3501, 5, 0), (9, 2, 0, 703, 1, 0), (32, 6, 0, 130, 3, 1), (40, 10, 0, 3103, 3, 0), (60, 15, 0, 61, 2, 0),
        (12, 0, 1, 90, 4, 0)]


def _jobs(dev, stream, spec):
    rec = synth.receptor(1200, 23)
    xyz, ty = torch.from_numpy(rec.xyz).to(dev), torch.from_numpy(rec.xs_type).to(dev)
    box = dsdp.make_box(rec.pocket_center, BOX, H)
    n = [int(np.ceil(BOX / H))] * 3
    keep, jobs, maps = [xyz, ty], [], {}
    for dtype in {s[2] for s in spec}:
        nb = dsdp.dsdp_grid_map_bytes(box, dtype)
        maps[dtype] = torch.empty(nb, dtype=torch.uint8, device=dev)
        dsdp.dsdp_grid_build_device(len(ty), xyz.data_ptr(), ty.data_ptr(), box, dtype, 0, maps[dtype].data_ptr(), nb,
                                    stream)
    for i, (atoms, T, dtype, chains, steps, opt) in enumerate(spec):
        lig = synth.ligand(atoms, T, 90 + i, center=rec.pocket_center)
        blob = dsdp.dsdp_ligand_pack(lig)
        nx = 7 + lig.n_torsions
        out = dict(conf=torch.zeros((chains, nx), device=dev), e=torch.zeros(chains, device=dev),
                   evals=torch.zeros(chains, dtype=torch.int32, device=dev),
                   trace=torch.zeros((chains, steps + 1, nx + 4), device=dev),
                   top=torch.zeros(9, dtype=torch.int32, device=dev), n=torch.zeros(1, dtype=torch.int32, device=dev),
                   score=torch.zeros(9, dtype=torch.float64, device=dev))
        d_blob = torch.from_numpy(blob).to(dev)
        j = dsdp.dsdp_job_device()
        j.grid = dsdp.grid_view(maps[dtype].data_ptr(), n, [c - (n[0] - 1) * H / 2 for c in rec.pocket_center], H, dtype)
        j.receptor = dsdp.dsdp_receptor(len(ty), xyz.data_ptr(), ty.data_ptr())
        j.h_blob, j.d_blob = blob.ctypes.data, d_blob.data_ptr()
        j.params = dsdp.make_params(n_chains=chains, n_mc_steps=steps, n_opt_iters=6, seed=i, optimizer=opt, trace=1)
        for a in range(3):
            j.box_lo[a], j.box_size[a] = rec.pocket_center[a] - BOX / 2, BOX
        j.d_chain_best_conf, j.d_chain_best_e = out["conf"].data_ptr(), out["e"].data_ptr()
        j.d_chain_evals, j.d_trace = out["evals"].data_ptr(), out["trace"].data_ptr()
        j.d_out_n, j.d_out_chain, j.d_out_score = out["n"].data_ptr(), out["top"].data_ptr(), out["score"].data_ptr()
        jobs.append(j)
        keep.append((blob, d_blob, out))
    return jobs, keep, [k[2] for k in keep[2:]], maps


def _take(outs):
    torch.cuda.synchronize()
    got = [{k: v.cpu().numpy().copy() for k, v in o.items()} for o in outs]
    for o in outs:
        for v in o.values():
            v.zero_()
    torch.cuda.synchronize()
    return got


@pytest.mark.parametrize("spec,graph", [(JOBS, False), (JOBS, True), (FEW[0], False), (FEW[1], False), (FEW[1], True)])
def test_sliced_chains_are_the_whole_chains(spec, graph):
    dev = torch.device("cuda", 0)
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        stream = side.cuda_stream
        jobs, keep, outs, maps = _jobs(dev, stream, spec)
        plan = dsdp.dsdp_plan_create(None, jobs, 0, 1)  # 128 registers, one chain per CTA, no queue
        dsdp.dsdp_plan_launch(plan, stream)
        want = _take(outs)
        dsdp.dsdp_plan_destroy(None, plan)
        assert all(w["evals"].min() > 0 for w in want)
        configs = [(0, 0), (0, 2), (1, 5), (1, 10)]  # automatic; queue with 1, 2 and 4 chains per CTA
        for flag, tile_config in configs[:1] if graph else configs:
            plan = dsdp.dsdp_plan_create(None, jobs, dsdp.DSDP_PLAN_PERSISTENT * flag, tile_config)
            if graph:
                g = torch.cuda.CUDAGraph()
                dsdp.dsdp_plan_launch(plan, stream)
                _take(outs)
                with torch.cuda.graph(g, stream=side):
                    dsdp.dsdp_plan_launch(plan, stream)
            for _ in range(2):
                if graph:
                    g.replay()
                else:
                    dsdp.dsdp_plan_launch(plan, stream)
                for w, o in zip(want, _take(outs)):
                    for k in w:
                        assert np.array_equal(w[k], o[k]), (tile_config, flag, k)
            if graph:
                del g
            dsdp.dsdp_plan_destroy(None, plan)
