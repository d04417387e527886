"""Edges of the grid, voxel and rescoring kernels' dispatch rules and tiles: brick
sizes, more kept atoms than one staging holds, atoms that are not at a finite
place, cell lists against the scan of every atom, part-filled tiles."""
import numpy as np
import pytest

import oracle
from paper_2303_09916_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2303_09916_gb300 import dsdp  # noqa: E402

DEV = "cuda"


def _maps(xyz, types, center, n, h, dtype=dsdp.DSDP_MAP_F32, mode=dsdp.DSDP_GRID_EQ4):
    box = dsdp.make_box(center, [k * h for k in n], h)
    d_xyz, d_ty = torch.from_numpy(np.ascontiguousarray(xyz, np.float32)).to(DEV), torch.from_numpy(types).to(DEV)
    ch, td = 4 if mode == dsdp.DSDP_GRID_EQ4 else 1, [torch.float32, torch.bfloat16, torch.float16][dtype]
    maps = torch.full((8, n[2], n[1], n[0], ch), float("nan"), dtype=td, device=DEV)
    dsdp.dsdp_grid_build_device(len(types), d_xyz.data_ptr(), d_ty.data_ptr(), box, dtype, mode, maps.data_ptr(),
                                maps.numel() * maps.element_size(), torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    return maps.float().cpu().numpy().astype(np.float64)


def test_grid_of_two_block_bricks_matches_the_small_grid():
    """107 x 110 x 104 vertices run two blocks a warp, the 9 x 11 x 13 grid of some of
    the same vertices (a power-of-two spacing: the same FP32 positions) one.  Both sum
    the same terms, in another order and some of them in another of the three forms:
    2e-6 of the values or of 10.  The other map types and kinds are that build's values,
    rounded."""
    rec = synth.receptor(3000, 5)
    h, n, m, off = 0.25, (107, 110, 104), (9, 11, 13), (40, 51, 47)
    origin = np.round(rec.pocket_center * 4) / 4 - 13.0
    center = [origin[a] + (n[a] - 1) * h / 2 for a in range(3)]
    wide = _maps(rec.xyz, rec.xs_type, center, n, h)
    small = _maps(rec.xyz, rec.xs_type, [origin[a] + (off[a] + (m[a] - 1) / 2) * h for a in range(3)], m, h)
    cut = wide[:, off[2]:off[2] + m[2], off[1]:off[1] + m[1], off[0]:off[0] + m[0]]
    assert np.isfinite(wide).all()
    assert np.all(np.abs(cut - small) <= 2e-6 * np.maximum(np.abs(small), 10.0))
    for dtype, td in ((dsdp.DSDP_MAP_BF16, torch.bfloat16), (dsdp.DSDP_MAP_F16, torch.float16)):
        for mode in (dsdp.DSDP_GRID_EQ4, dsdp.DSDP_GRID_EQ3):
            want = torch.from_numpy(wide[..., : 4 if mode == dsdp.DSDP_GRID_EQ4 else 1]).float().to(td).double().numpy()
            assert np.array_equal(_maps(rec.xyz, rec.xs_type, center, n, h, dtype, mode), want)


def test_grid_with_more_atoms_in_reach_than_one_staging_holds():
    """Maps add up over the receptor's atoms: 7,000 atoms in reach of every brick
    (staged 1,536 at a time) against the sum of seven maps of 1,000, to 1e-6 of the
    largest possible sum of the terms' magnitudes (12.2 and 6.4 an atom).  Atoms at
    NaN and infinite places change nothing."""
    rng = np.random.default_rng(3)
    xyz = rng.uniform(-6, 6, (7000, 3)).astype(np.float32)
    types = rng.integers(0, 9, 7000).astype(np.uint8)
    n, h = (11, 9, 5), 0.375
    whole = _maps(xyz, types, [0.1, 0.2, 0.3], n, h)
    parts = sum(_maps(xyz[k::7], types[k::7], [0.1, 0.2, 0.3], n, h) for k in range(7))
    assert np.abs(whole[..., 0] - parts[..., 0]).max() <= 1e-6 * 7000 * 12.2
    assert np.abs(whole[..., 1:] - parts[..., 1:]).max() <= 1e-6 * 7000 * 6.4
    bad = np.array([[np.nan, 0, 0], [0, np.inf, 0], [0, -np.inf, np.nan]], np.float32)
    again = _maps(np.concatenate([xyz, bad]), np.concatenate([types, types[:3]]), [0.1, 0.2, 0.3], n, h)
    assert np.array_equal(whole, again)


def _voxels(xyz, radius, feats, center):
    d = [torch.from_numpy(np.ascontiguousarray(a, np.float32)).to(DEV) for a in (xyz, radius, feats)]
    out = torch.full((36, 36, 36, 18), -1.0, device=DEV)
    work = torch.full((dsdp.dsdp_voxel_work_bytes() + 8,), 0xA5, dtype=torch.uint8, device=DEV)
    dsdp.dsdp_voxelize_device(len(radius), *[t.data_ptr() for t in d], center, out.data_ptr(), work.data_ptr() + 8,
                              work.numel() - 8, torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    return out.cpu().numpy()


@pytest.mark.parametrize("case", ["plain", "large_radii", "odd_values"])
def test_voxel_cell_lists_match_the_scan_of_every_atom(case):
    """The same atoms with 170,000 more far outside the cube (too many for cell lists:
    every atom is scanned) give the same bits: atoms on all sides of the cube's faces,
    radii that reach over several cells, radii and places that are not finite."""
    rng = np.random.default_rng(7)
    xyz = rng.uniform(-42, 42, (900, 3))
    radius, feats = rng.uniform(1.2, 2.0, 900), rng.uniform(-1, 1, (900, 17))
    feats[::3] = np.round(feats[::3])
    if case == "large_radii":
        radius[::50] = rng.uniform(8, 20, 18)
    if case == "odd_values":
        radius[:4] = [-9.0, np.nan, -1.4, 0.0]
        xyz[4], xyz[5] = [np.nan, 0, 0], [np.inf, 0, 0]
        xyz[6:40] = xyz[40:74]  # atoms at the same place
    far = np.concatenate([xyz, rng.uniform(500, 600, (170000, 3))])
    one = _voxels(xyz, radius, feats, [0.5, -0.25, 1.0])
    all_ = _voxels(far, np.concatenate([radius, np.full(170000, 1.7)]), np.concatenate([feats, np.ones((170000, 17))]),
                   [0.5, -0.25, 1.0])
    assert one[..., 17].sum() > 0
    assert np.array_equal(one, all_)


@pytest.mark.parametrize("n_rec,n_chains,atoms,T", [(1, 1, 5, 0), (512, 9, 33, 6), (513, 7, 64, 15), (1500, 18, 20, 4)])
def test_rescoring_of_part_filled_tiles_matches_the_oracle(n_rec, n_chains, atoms, T):
    rec = synth.receptor(max(n_rec, 300), 8)
    xyz, types = rec.xyz[-n_rec:], rec.xs_type[-n_rec:]
    lig = synth.ligand(atoms, T, 9, center=xyz.astype(np.float64).mean(0))
    olig = oracle.Ligand(lig.xyz.astype(np.float64), lig.xs_type, lig.bonds, lig.rotatable)
    rng = np.random.default_rng(n_rec)
    conf = np.tile(olig.identity_conf(), (n_chains, 1))
    conf[:, :3] += rng.uniform(-4, 4, (n_chains, 3))
    conf[:, 3:7] = rng.normal(size=(n_chains, 4))
    conf[:, 7:] = rng.uniform(-3, 3, (n_chains, lig.n_torsions))
    conf = conf.astype(np.float32)
    blob = dsdp.dsdp_ligand_pack(lig)
    d = [torch.from_numpy(np.ascontiguousarray(a)).to(DEV) for a in (xyz, types, blob, conf)]
    out = dict(n=torch.zeros(1, dtype=torch.int32, device=DEV), chain=torch.zeros(9, dtype=torch.int32, device=DEV),
               score=torch.zeros(9, dtype=torch.float64, device=DEV), intra=torch.zeros(9, dtype=torch.float64, device=DEV))
    j = dsdp.dsdp_job_device()
    j.receptor = dsdp.dsdp_receptor(n_rec, d[0].data_ptr(), d[1].data_ptr())
    j.h_blob, j.d_blob, j.d_chain_best_conf = blob.ctypes.data, d[2].data_ptr(), d[3].data_ptr()
    j.params = dsdp.make_params(n_chains=n_chains, top_k=9)
    j.d_out_n, j.d_out_chain = out["n"].data_ptr(), out["chain"].data_ptr()
    j.d_out_score, j.d_out_intra = out["score"].data_ptr(), out["intra"].data_ptr()
    dsdp.dsdp_rescore_topk_noalloc(j, torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    scores, idx, terms = oracle.rescore_topk(olig, xyz.astype(np.float64), types, conf.astype(np.float64), k=9)
    k = int(out["n"].item())
    assert k == len(idx) and out["chain"][:k].tolist() == list(idx)
    assert np.allclose(out["score"][:k].cpu().numpy(), terms[:, 0], rtol=1e-10, atol=1e-10)
    assert np.allclose(out["intra"][:k].cpu().numpy(), terms[:, 2], rtol=1e-10, atol=1e-10)
