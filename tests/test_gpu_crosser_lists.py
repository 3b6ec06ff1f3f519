"""Crossers past their queues while the spill list is nearly full: rows of a tile crowded beyond their
slots and hot, so that the share of the queue of the CTAs that own these rows overflows.  Neither list
takes the other's room, and the run has the bits of one with room for all."""
import dataclasses

import numpy as np
import pytest

import pic_inputs as pi

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pic():
    import __graft_entry__ as ge
    ge.build()
    import paper_0808_4078_gb300 as pic
    return pic


def _striped(nx, ny, rows, ppc, nu):
    """Particles in the first `rows` of every 16 rows."""
    wl = pi.weibel_load(ndim=2, nx=nx, ny=ny, ppc=ppc, T_perp_beam=1.1, T_bg=0.12, nu=nu, seed=81)
    sp = []
    for s in wl.species:
        k = (s.cell // nx) % 16 < rows
        sp.append(dataclasses.replace(s, cell=s.cell[k], offset=s.offset[:, k], u=s.u[:, k]))
    return dataclasses.replace(wl, species=sp)


# 245760 particles per species, 49152 of them past their cells' slots and 65536 places for these; the
# hot rows' CTAs leave another ~50000.  Small grid: a CTA per row; 320 tiles: four rows per CTA
@pytest.mark.parametrize("nx,ny,rows,ppc,cc", [(64, 64, 6, 160, 128), (320, 256, 4, 24, 20)])
def test_queue_overflow_beside_a_full_spill_list(pic, nx, ny, rows, ppc, cc):
    wl = _striped(nx, ny, rows, ppc, 0.1)
    out = []
    for cap in (cc, 4 * ppc):
        eng = pic.Engine.from_workload(wl, track_ids=True, diag_interval=1, diag_capacity=8, cell_capacity=(cap, cap))
        eng.step(3)
        eng.sync()
        res = list(eng.fields()[:2])
        for s in range(2):
            cell, off, u, ids = eng.particles(s)
            o = np.argsort(ids)
            res += [cell[o], off[:, o], u[:, o]]
        recs = eng.diag()
        res += [np.array([[r["Ekin"][0], r["Ekin"][1], *r["P"]] for r in recs])]
        out.append(res)
        eng.close()
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)
