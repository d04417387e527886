"""What the autotuner records is for plans that it says something about."""
import numpy as np
import pytest

from paper_2303_09916_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2303_09916_gb300 import dsdp  # noqa: E402

from graph_nodes import captured_kernels  # noqa: E402

BOX, H = 9.0, 0.375


@pytest.fixture(scope="module")
def jobs():
    """make(chains, optimizer, atoms): one job on FP16 Eq. 3 maps (no other test tunes plans of these)."""
    rec = synth.receptor(300, 4)
    side = torch.cuda.Stream()
    xyz, ty = torch.from_numpy(rec.xyz).cuda(), torch.from_numpy(rec.xs_type).cuda()
    box, n = dsdp.make_box(rec.pocket_center, BOX, H), int(np.ceil(BOX / H))
    nb = dsdp.dsdp_grid_map_bytes(box, dsdp.DSDP_MAP_F16, dsdp.DSDP_GRID_EQ3)
    maps = torch.empty(nb, dtype=torch.uint8, device="cuda")
    dsdp.dsdp_grid_build_device(len(ty), xyz.data_ptr(), ty.data_ptr(), box, dsdp.DSDP_MAP_F16, dsdp.DSDP_GRID_EQ3,
                                maps.data_ptr(), nb, torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    keep = [maps, xyz, ty]

    def make(chains, optimizer, atoms=12, steps=2):
        lig = synth.ligand(atoms, 2, 5, center=rec.pocket_center)
        blob = dsdp.dsdp_ligand_pack(lig)
        d_blob = torch.from_numpy(blob).cuda()
        j = dsdp.dsdp_job_device()
        j.grid = dsdp.grid_view(maps.data_ptr(), [n] * 3, [c - (n - 1) * H / 2 for c in rec.pocket_center], H,
                                dsdp.DSDP_MAP_F16, dsdp.DSDP_GRID_EQ3)
        j.h_blob, j.d_blob = blob.ctypes.data, d_blob.data_ptr()
        j.params = dsdp.make_params(n_chains=chains, n_mc_steps=steps, n_opt_iters=8, seed=2, optimizer=optimizer)
        for a in range(3):
            j.box_lo[a], j.box_size[a] = rec.pocket_center[a] - BOX / 2, BOX
        keep.extend([blob, d_blob])
        return [j]

    return make, side.cuda_stream, keep + [side]


def _create(jobs, tile_config=0):
    return dsdp.dsdp_plan_create(None, jobs, dsdp.DSDP_PLAN_NO_RESCORE, tile_config)


def test_tuning_one_optimiser_leaves_the_other_its_teams(jobs):
    make, stream, _ = jobs
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    chains = 2 * sms
    before, after = [], []
    for seen in (before, after):
        plan = _create(make(chains, dsdp.DSDP_OPT_BFGS))
        seen += captured_kernels(stream, lambda: dsdp.dsdp_plan_launch(plan, stream))
        dsdp.dsdp_plan_destroy(None, plan)
        if seen is before:  # Barzilai-Borwein: no line search, no teams, always a fixed choice
            plan = _create(make(chains, dsdp.DSDP_OPT_BB))
            dsdp.dsdp_plan_autotune(plan, stream, 1)
            dsdp.dsdp_plan_destroy(None, plan)
    assert before == [(chains, 4 * 32)] and after == before


def test_tuning_measures_the_automatic_arrangement_of_every_plan(jobs):
    """A plan created with a fixed choice: teams of four take less than half of what the best
    fixed configuration does, so tuning leaves the plan with them and later plans too, also
    where an earlier record of the shape had taken them away."""
    make, stream, _ = jobs
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    chains = 2 * sms
    for tile_config in (1, 0):
        plan = _create(make(chains, dsdp.DSDP_OPT_BFGS, steps=12), tile_config)
        dsdp.dsdp_plan_autotune(plan, stream, 3)
        assert captured_kernels(stream, lambda: dsdp.dsdp_plan_launch(plan, stream)) == [(chains, 4 * 32)]
        dsdp.dsdp_plan_destroy(None, plan)
        plan = _create(make(chains, dsdp.DSDP_OPT_BFGS))
        assert captured_kernels(stream, lambda: dsdp.dsdp_plan_launch(plan, stream)) == [(chains, 4 * 32)]
        dsdp.dsdp_plan_destroy(None, plan)


@pytest.mark.parametrize("chains_per_sm,optimizer", [(0.5, 0), (2, 0), (12, 0), (2, 1), (12, 1), (40, 0)])
def test_a_plan_made_from_the_kept_configuration_runs_what_the_tuned_plan_runs(jobs, chains_per_sm, optimizer):
    make, stream, _ = jobs
    chains = int(chains_per_sm * torch.cuda.get_device_properties(0).multi_processor_count)
    spec = make(chains, optimizer, steps=6)
    plan = _create(spec)
    kept = dsdp.dsdp_plan_config(plan)  # before: the automatic arrangement, or the fixed one that it is
    runs = captured_kernels(stream, lambda: dsdp.dsdp_plan_launch(plan, stream))
    again = _create(spec, 1 + (kept - 1) % 12 if kept else 0)
    assert captured_kernels(stream, lambda: dsdp.dsdp_plan_launch(again, stream)) == runs
    dsdp.dsdp_plan_destroy(None, again)
    chosen, ms = dsdp.dsdp_plan_autotune(plan, stream, 2, with_times=True)
    kept = dsdp.dsdp_plan_config(plan)
    assert kept in (0, chosen) and ms[chosen] == min(ms.values())
    again = dsdp.dsdp_plan_create(None, spec, dsdp.DSDP_PLAN_NO_RESCORE | (dsdp.DSDP_PLAN_PERSISTENT if kept > 12 else 0),
                                  1 + (kept - 1) % 12 if kept else 0)
    assert dsdp.dsdp_plan_config(again) == kept
    assert dsdp.dsdp_plan_kernel_count(again) == dsdp.dsdp_plan_kernel_count(plan)
    runs = [captured_kernels(stream, lambda: dsdp.dsdp_plan_launch(p, stream)) for p in (plan, again)]
    assert runs[0] == runs[1] and len(runs[0]) == dsdp.dsdp_plan_kernel_count(plan)
    for p in (plan, again):
        dsdp.dsdp_plan_destroy(None, p)
