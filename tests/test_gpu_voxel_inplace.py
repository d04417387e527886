"""Voxel features written over their own inputs (the output replaces an array that is
not needed any more)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2303_09916_gb300 import dsdp  # noqa: E402


@pytest.mark.parametrize("shared", ["xyz", "radius", "features"])
@pytest.mark.parametrize("place", ["start", "end"])
def test_output_over_an_input_gives_the_same_voxels(shared, place):
    rng = np.random.default_rng(4)
    n = 500
    arrays = dict(xyz=rng.uniform(-30, 30, (n, 3)), radius=rng.uniform(1.2, 2.0, n),
                  features=rng.uniform(-1, 1, (n, 17)))
    size, got = 36 * 36 * 36 * 18, []
    work = torch.empty(dsdp.dsdp_voxel_work_bytes(), dtype=torch.uint8, device="cuda")
    for over in (False, True):
        d = {k: torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda().flatten() for k, a in arrays.items()}
        m = d[shared].numel()
        # the input at the output's first values, or half of it beyond its last ones
        at = 0 if place == "start" else size - m // 2
        buf = torch.full((size + m,), 7.0, device="cuda")
        buf[at:at + m] = d[shared]
        if over:
            d[shared] = buf[at:at + m]
        torch.cuda.synchronize()
        dsdp.dsdp_voxelize_device(n, *[d[k].data_ptr() for k in ("xyz", "radius", "features")], [0.3, 0.1, -0.2],
                                  buf.data_ptr(), work.data_ptr(), work.numel(), torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        got.append(buf[:size].cpu().numpy())
    assert got[0].reshape(-1, 18)[:, 17].sum() > 0
    assert np.array_equal(got[0], got[1])
