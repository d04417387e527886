"""The distance that the far atoms' Gaussian is evaluated at, for every pair of radii."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2303_09916_gb300 import dsdp  # noqa: E402

RADII = {1.9: 0, 1.8: 2, 1.7: 5, 2.0: 7}  # and a type of each


def test_far_atoms_distance_is_rounded_alike_for_all_radii():
    """One atom, 6.6 to 7.8 A away: a map is W exp(-b^2), b = (r - R - s - 3) / 2, and its
    relative error's slope against 2 b is the constant error of b, of which the radii's
    part is what differs between the pairs of radii.  The offset of a pair is rounded
    once, at below 1 in units of b / 1.2: 6e-8 between any two, and 4e-8 for the other
    roundings, which vary from vertex to vertex (1.5e-7 in 9,216 vertices)."""
    h, n = 1.0 / 32, (24, 24, 16)
    center = np.array([4.0, 4.25, 4.125])
    box = dsdp.make_box(center + h / 2, [k * h for k in n], h)
    axes = [center[a] + h / 2 - (n[a] - 1) * h / 2 + h * np.arange(n[a]) for a in range(3)]
    z, y, x = np.meshgrid(axes[2], axes[1], axes[0], indexing="ij")
    r = np.sqrt(x * x + y * y + z * z)
    assert 6.45 < r.min() and r.max() < 7.95
    xyz = torch.zeros(3, device="cuda")
    off = []
    for R, tj in RADII.items():
        ty = torch.tensor([tj], dtype=torch.uint8, device="cuda")
        maps = torch.empty((8, n[2], n[1], n[0], 4), device="cuda")
        dsdp.dsdp_grid_build_device(1, xyz.data_ptr(), ty.data_ptr(), box, dsdp.DSDP_MAP_F32, dsdp.DSDP_GRID_EQ4,
                                    maps.data_ptr(), maps.numel() * 4, torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        got = maps[..., 0].double().cpu().numpy()
        for s, t in RADII.items():
            b = 0.5 * (r - R - s - 3.0)
            want = -0.00516 * np.exp(-b * b) - 0.0356 * np.exp(-4.0 * (r - R - s) ** 2)
            off.append(-np.polyfit((2.0 * b).ravel(), (got[t] / want - 1.0).ravel(), 1)[0])
    off = np.array(off) * 1.2
    assert off.max() - off.min() <= 1e-7, off
