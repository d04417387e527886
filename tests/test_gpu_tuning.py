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


def test_plans_in_flight_share_the_gpu_without_teams(jobs):
    """The way of a plan's chains goes by all chains under way at its launch: two plans of 8
    chains per SM each run for long on two streams; a third plan's teams then stay while
    one of them counts (its own stream's launches come before it) and go with both."""
    make, stream, _ = jobs
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    torch.cuda.synchronize()
    side = [torch.cuda.Stream() for _ in range(3)]
    long_ = [_create(make(8 * sms + k, 0, atoms=30, steps=600), 1) for k in range(2)]
    ends = [torch.cuda.Event() for _ in long_]
    small, tiny, other = _create(make(2 * sms, 0)), _create(make(sms, 0)), _create(make(2 * sms, 0))
    seen = []

    def launch(plan, st):
        dsdp.dsdp_plan_launch(plan, st.cuda_stream)
        seen.append(dsdp.dsdp_plan_team(plan))

    assert dsdp.dsdp_plan_team(small) == 0
    launch(small, side[2])
    launch(tiny, side[2])
    torch.cuda.synchronize()
    assert seen == [4, 8]
    dsdp.dsdp_plan_launch(long_[0], side[0].cuda_stream)
    ends[0].record(side[0])
    launch(tiny, side[2])  # 9 per SM
    launch(small, side[2])  # 10
    dsdp.dsdp_plan_launch(long_[1], side[1].cuda_stream)
    ends[1].record(side[1])
    launch(small, side[2])  # 18
    launch(other, side[1])  # 10 to 12 beside its own stream's
    under_way = not any(e.query() for e in ends)
    assert captured_kernels(stream, lambda: dsdp.dsdp_plan_launch(small, stream)) == [(2 * sms, 4 * 32)]
    torch.cuda.synchronize()
    launch(small, side[2])
    torch.cuda.synchronize()
    launch(tiny, side[1])
    torch.cuda.synchronize()
    assert under_way and seen[2:] == [4, 4, 1, 4, 4, 8]
    for p in [*long_, small, tiny, other]:
        dsdp.dsdp_plan_destroy(None, p)
