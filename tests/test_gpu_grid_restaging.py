"""Two blocks of vertices a warp and more atoms in reach than one staging holds: the
second block reads the receptor again."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from gpu_util import E_REL  # noqa: E402
from test_gpu_kernel_edges import _maps  # noqa: E402


@pytest.mark.parametrize("atoms", [1536, 1537, 4100])
def test_second_block_of_a_brick_stages_the_receptor_again(atoms):
    """All atoms within 3 A of the middle, in reach of every brick there: vertices of both
    blocks of the bricks around it against the oracle, energies to 1e-4 of the sum of the
    terms' magnitudes (an atom left out of a staging is more than that on most)."""
    rng = np.random.default_rng(atoms)
    xyz = rng.uniform(-3, 3, (atoms, 3)).astype(np.float32)
    types = rng.integers(0, 9, atoms).astype(np.uint8)
    n, h, center = (107, 110, 104), 0.25, np.array([0.05, -0.1, 0.2])
    maps = _maps(xyz, types, center, n, h)
    assert np.isfinite(maps).all()
    at = [rng.integers(n[a] // 2 - 12, n[a] // 2 + 12, 1500) for a in range(3)]
    pts = np.stack([center[a] + (at[a] - (n[a] - 1) / 2) * h for a in range(3)], -1)
    assert set((at[2] // 4) % 2) == {0, 1}
    x64 = xyz.astype(np.float64)
    for t in range(8):
        want = oracle.receptor_field(x64, types, t, pts)[:, 0]
        scale = oracle.receptor_field_abs(x64, types, t, pts)[:, 0]
        err = np.abs(maps[t, at[2], at[1], at[0], 0] - want)
        assert np.all(err <= E_REL * np.maximum(scale, 1.0)), (t, (err / scale).max())
