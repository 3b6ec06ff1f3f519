"""Small grids share each tile among 8 or 16 CTAs, large ones among 4; the same run inside a batch
with a large one takes the large grids' split.  Both are the same bits (integer
deposits, the same per-particle operations, the field energies summed per tile)."""
import numpy as np
import pytest

import pic_inputs

pytestmark = pytest.mark.gpu


def _state(eng, run):
    out = [np.array([[r["WE"], r["WB"], r["P"]] for r in eng.diag(run=run)]),
           np.array([r["Ekin"] for r in eng.diag(run=run)]), *eng.fields(run=run)[:2]]
    for s in range(2):
        cell, off, u, ids = eng.particles(s, run=run)
        o = np.argsort(ids)
        out += [cell[o], off[:, o], u[:, o]]
    return out


# 4, 36, 40, 76, 88, 152 tiles: 16, 16, 8, 8, 8, 8 parts per tile
@pytest.mark.parametrize("tile", [(16, 16), (32, 8), (8, 32)])
@pytest.mark.parametrize("nx,ny,ppc", [(32, 32, 3), (96, 96, 33), (160, 64, 8), (608, 32, 5), (352, 64, 9),
                                       (1216, 32, 4)])
def test_small_grid_equals_the_run_in_a_large_batch(nx, ny, ppc, tile):
    import paper_0808_4078_gb300 as pic
    # the hot beam of odd counts crosses cells faster than its queue holds
    T = 8.0 if ppc % 2 else 0.5
    small = pic_inputs.weibel_load(ndim=2, nx=nx, ny=ny, ppc=ppc, T_perp_beam=T, T_bg=0.05, nu=0.2, seed=9)
    large = pic_inputs.weibel_load(ndim=2, nx=320, ny=320, ppc=4, T_perp_beam=0.1, seed=10)
    kw = dict(track_ids=True, diag_interval=1, diag_capacity=32, tile=tile, cell_capacity=(256, 256))
    alone = pic.Engine.from_workloads([small], **kw)
    batch = pic.Engine.from_workloads([small, large], **kw)
    for eng in (alone, batch):
        eng.step(12)
        eng.sync()
    for a, b in zip(_state(alone, 0), _state(batch, 0)):
        np.testing.assert_array_equal(a, b)
    if nx * ny <= 1024:
        import oracle
        sim = oracle.Simulation.from_workload(small)
        sim.step(12)
        for s in range(2):
            uo = sim.species[s].u
            assert np.abs(_state(alone, 0)[6 + 3 * s].astype(np.float64) - uo).max() < 1e-4 * np.abs(uo).max()
    alone.close()
    batch.close()
