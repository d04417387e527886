"""Ligands of a few atoms in the job queue."""
import numpy as np
import pytest

from paper_2303_09916_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2303_09916_gb300 import dsdp  # noqa: E402


@pytest.mark.parametrize("atoms,torsions", [(2, 0), (4, 0), (5, 1)])
def test_small_ligand_fits_the_budget_of_its_coordinates(atoms, torsions):
    """8,192 chains need about 150 + 24 atoms bytes each beside their results: 2.6 MB
    are enough for them (the time-sliced queue, which they take, keeps a record per
    chain in the same memory), and all chains are searched."""
    rec = synth.receptor(300, 3)
    ctx = dsdp.dsdp_create(0, mem_budget_bytes=2600000)
    try:
        grid = dsdp.dsdp_grid_build(ctx, rec.xyz, rec.xs_type, dsdp.make_box(rec.pocket_center, 6.0, 0.5), 0)
        try:
            lig = synth.ligand(atoms, torsions, 2, center=rec.pocket_center)
            p = dsdp.make_params(n_chains=8192, n_mc_steps=2, n_opt_iters=4, seed=3)
            job = dsdp.dsdp_dock_submit_many(ctx, [grid], [lig], [p])[0]
            r = dsdp.dsdp_dock_poll(ctx, job, dsdp.result_buffers(lig.n_atoms, lig.n_torsions, p), -1)
            assert r["n_out"] >= 1 and np.isfinite(r["score"][: r["n_out"]]).all()
            assert len(r["chain_best_e"]) == 8192 and np.isfinite(r["chain_best_e"]).all()
            assert len(np.unique(r["chain_best_e"])) > 100
        finally:
            dsdp.dsdp_grid_free(ctx, grid)
    finally:
        dsdp.dsdp_destroy(ctx)
