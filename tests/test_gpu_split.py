"""The shared-memory split that a chain launch asks for, by the maps it reads."""
import pytest

from paper_2303_09916_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2303_09916_gb300 import dsdp  # noqa: E402

from graph_nodes import CARVEOUT, captured_kernels  # noqa: E402


@pytest.mark.parametrize("n_maps,atoms,optimizer,percent", [(1, 30, 0, 73), (2, 30, 0, 59), (2, 30, 1, 73), (2, 40, 0, None)])
def test_split_by_the_size_of_the_maps(n_maps, atoms, optimizer, percent):
    """Maps of 432 MB each (nothing is launched on them): one is below 4 times the L2 cache,
    two are above, which the optimiser without a line search does not mind; ligands of more
    than 32 atoms do not ask."""
    l2 = torch.cuda.get_device_properties(0).L2_cache_size
    assert 432e6 <= 4 * l2 < 864e6
    buf = torch.zeros(64, device="cuda")
    lig = synth.ligand(atoms, 6, 5, center=[0.0, 0.0, 0.0])
    blob = dsdp.dsdp_ligand_pack(lig)
    d_blob = torch.from_numpy(blob).cuda()
    jobs = []
    for k in range(4):
        j = dsdp.dsdp_job_device()
        j.grid = dsdp.grid_view(buf.data_ptr() + 16 * (k % n_maps), [150] * 3, [0.0] * 3, 0.375)
        j.h_blob, j.d_blob = blob.ctypes.data, d_blob.data_ptr()
        j.params = dsdp.make_params(n_chains=1000, n_mc_steps=4, seed=k, optimizer=optimizer)
        for a in range(3):
            j.box_size[a] = 10.0
        jobs.append(j)
    stream = torch.cuda.Stream()
    plan = dsdp.dsdp_plan_create(None, jobs, dsdp.DSDP_PLAN_NO_RESCORE, 0)
    got = captured_kernels(stream.cuda_stream, lambda: dsdp.dsdp_plan_launch(plan, stream.cuda_stream), CARVEOUT)
    assert got[0] == percent if percent else got[0] not in (59, 73)
    dsdp.dsdp_plan_destroy(None, plan)
