"""Launches of one kernel by several host threads with different shared-memory sizes."""
import threading

import numpy as np
import pytest

from paper_2303_09916_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2303_09916_gb300 import dsdp  # noqa: E402


def _rescoring_plan(n_chains, rec, dev):
    """A job whose ranking takes 12 bytes of shared memory per chain (a power of two)."""
    lig = synth.ligand(9, 1, 4, center=rec.pocket_center)
    blob = dsdp.dsdp_ligand_pack(lig)
    xyz, ty = torch.from_numpy(rec.xyz).to(dev), torch.from_numpy(rec.xs_type).to(dev)
    node = torch.zeros(8 * 8 * 4, device=dev)
    conf = torch.zeros((n_chains, 7 + lig.n_torsions), device=dev)
    conf[:, :3] = torch.from_numpy(np.asarray(rec.pocket_center, np.float32)).to(dev)
    conf[:, 3] = 1.0
    n_out, d_blob = torch.zeros(1, dtype=torch.int32, device=dev), torch.from_numpy(blob).to(dev)
    j = dsdp.dsdp_job_device()
    j.grid = dsdp.grid_view(node.data_ptr(), [2] * 3, rec.pocket_center, 0.375)
    j.receptor = dsdp.dsdp_receptor(len(ty), xyz.data_ptr(), ty.data_ptr())
    j.h_blob, j.d_blob = blob.ctypes.data, d_blob.data_ptr()
    j.params = dsdp.make_params(n_chains=n_chains, n_mc_steps=1, n_opt_iters=1, seed=1)
    j.d_chain_best_conf, j.d_out_n = conf.data_ptr(), n_out.data_ptr()
    return dsdp.dsdp_plan_create(None, [j], 0, 1), n_out, (blob, xyz, ty, node, conf, d_blob, j)


def test_threads_with_different_shared_memory():
    """8,192 and 4,096 chains rank in 96 and 48 KB: neither thread's launches may be
    refused because the other has just asked for its own size."""
    dev = torch.device("cuda", 0)
    rec = synth.receptor(40, 5)
    plans = [_rescoring_plan(n, rec, dev) for n in (8192, 4096)]
    torch.cuda.synchronize()
    start, errors, streams = threading.Barrier(2), [], [torch.cuda.Stream() for _ in plans]

    def work(k):
        start.wait()
        try:
            for _ in range(400):
                dsdp.dsdp_plan_launch_stage(plans[k][0], dsdp.DSDP_STAGE_RESCORE, streams[k].cuda_stream)
        except Exception as e:  # a refused launch
            errors.append((k, str(e)))

    threads = [threading.Thread(target=work, args=(k,)) for k in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    for plan, n_out, _ in plans:
        dsdp.dsdp_plan_destroy(None, plan)
        assert int(n_out.item()) == 1  # every pose is the same
    assert not errors, errors
