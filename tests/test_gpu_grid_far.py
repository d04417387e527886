"""Maps of receptors far from the origin, where FP32 coordinates are coarse."""
import numpy as np
import pytest

import oracle
from paper_2303_09916_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2303_09916_gb300 import dsdp  # noqa: E402


@pytest.mark.parametrize("place,n", [(3.0e4, (40, 33, 36)), (-2.2e5, (40, 33, 36)), (9.0e5, (40, 33, 36)),
                                     (2.2e5, (107, 110, 104))])
def test_maps_far_from_the_origin_match_the_oracle_at_the_fp32_vertices(place, n):
    """A vertex lies at the FP32 nearest to origin + h i.  Distances between FP32 points
    this far out are exact in FP32 (multiples of 1/512 to 1/16 A, squares of less than
    24 bits), so an atom is in range of a vertex or not without ambiguity; energies to 1e-4 of the
    terms' magnitudes, as for every map.  (Both block depths of the kernel.)"""
    rec = synth.receptor(1500, 6)
    h = 0.3
    shift = np.array([place, -0.7 * place, 0.4 * place])
    xyz = (rec.xyz.astype(np.float64) + shift).astype(np.float32)
    center = rec.pocket_center + shift
    box = dsdp.make_box(center, [(k - 0.5) * h for k in n], h)
    assert [int(np.ceil((k - 0.5) * h / h)) for k in n] == list(n)
    d_xyz, d_ty = torch.from_numpy(xyz).cuda(), torch.from_numpy(rec.xs_type).cuda()
    maps = torch.full((8, n[2], n[1], n[0], 4), float("nan"), device="cuda")
    dsdp.dsdp_grid_build_device(len(d_ty), d_xyz.data_ptr(), d_ty.data_ptr(), box, dsdp.DSDP_MAP_F32,
                                dsdp.DSDP_GRID_EQ4, maps.data_ptr(), maps.numel() * 4,
                                torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    got = maps[..., 0].double().cpu().numpy()
    axes = []
    for a in range(3):
        o = np.float64(np.float32(center[a] - (n[a] - 1) * h / 2.0))
        axes.append((o + np.float64(np.float32(h)) * np.arange(n[a])).astype(np.float32).astype(np.float64))
    rng = np.random.default_rng(1)  # a sample of the vertices
    at = [rng.integers(0, n[a], 4000) for a in range(3)]
    pts = np.stack([axes[a][at[a]] for a in range(3)], -1)
    x64 = xyz.astype(np.float64)
    for t in range(8):
        want = oracle.receptor_field(x64, rec.xs_type, t, pts)[:, 0]
        scale = oracle.receptor_field_abs(x64, rec.xs_type, t, pts)[:, 0]
        err = np.abs(got[t, at[2], at[1], at[0]] - want)
        assert np.all(err <= 1e-4 * np.maximum(scale, 1.0)), (t, err.max())
