"""A pose's score and gradient do not depend on the batch it is in: the kernel for
batches of up to four conformations per SM and the one for more give the same bits."""
import numpy as np
import pytest

from paper_2303_09916_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2303_09916_gb300 import dsdp  # noqa: E402

N, H = 40, 0.375  # vertices per axis; some atoms lie outside


@pytest.mark.parametrize("atoms,torsions", [(2, 0), (9, 2), (32, 9), (33, 9), (64, 15)])
def test_scores_do_not_depend_on_the_batch(atoms, torsions):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    small, large = 4 * sms, 4 * sms + 33
    rng, gen = np.random.default_rng(atoms), torch.Generator().manual_seed(atoms)
    lig = synth.ligand(atoms, torsions, 3, center=np.zeros(3))
    blob = dsdp.dsdp_ligand_pack(lig)
    nd = 6 + lig.n_torsions
    conf = np.empty((large, 1 + nd), np.float32)
    conf[:, :3] = rng.uniform(-6.0, 6.0, (large, 3))
    q = rng.normal(size=(large, 4))
    conf[:, 3:7] = q / np.linalg.norm(q, axis=1, keepdims=True)
    conf[:, 7:] = rng.uniform(-np.pi, np.pi, (large, nd - 6))
    d_conf, d_blob = torch.from_numpy(conf).cuda(), torch.from_numpy(blob).cuda()
    stream = torch.cuda.current_stream().cuda_stream
    for dtype, tdtype in enumerate((torch.float32, torch.bfloat16, torch.float16)):
        for mode in (dsdp.DSDP_GRID_EQ4, dsdp.DSDP_GRID_EQ3):
            maps = torch.randn((8, N, N, N, 4 if mode == 0 else 1), generator=gen).to(tdtype).cuda().contiguous()
            view = dsdp.grid_view(maps.data_ptr(), [N] * 3, [-(N - 1) * H / 2] * 3, H, dtype, mode)
            got = []
            for n in (small, large):
                e, g = torch.zeros(large, device="cuda"), torch.zeros((large, nd), device="cuda")
                dsdp.dsdp_score_eval_device(view, blob, d_blob.data_ptr(), d_conf.data_ptr(), n, e.data_ptr(),
                                            g.data_ptr(), dsdp.DSDP_TERM_ALL, stream)
                torch.cuda.synchronize()
                got.append((e[:small].cpu().numpy(), g[:small].cpu().numpy()))
            assert np.isfinite(got[0][0]).all() and np.abs(got[0][1]).max() > 0
            assert np.array_equal(got[0][0], got[1][0]) and np.array_equal(got[0][1], got[1][1]), (dtype, mode)
