"""Variants of the 2D particle kernel on grids that fill the GPU (more than 304 tiles): the three tile
shapes times three register budgets with 4 CTAs per tile, and the 2-part kernel of each shape that runs
of at most 17 particles per cell take, all bitwise equal; and both under the bounds-checked build."""
import json
import os
import subprocess
import sys

import numpy as np
import pytest

import pic_inputs as pi

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SHAPES = [(16, 16), (32, 8), (8, 32)]


@pytest.fixture(scope="module")
def pic():
    import __graft_entry__ as ge
    ge.build()
    import paper_0808_4078_gb300 as pic
    return pic


def _run(pic, wl, tile, ctas, steps):
    eng = pic.Engine.from_workload(wl, track_ids=True, sort_interval=4, flags=pic.PIC_FLAG_KEEP_J, tile=tile,
                                   ctas_per_sm=ctas, diag_capacity=16)
    eng.step(steps)
    out = list(eng.fields(with_J=True))
    for s in range(2):
        cell, off, u, ids = eng.particles(s)
        o = np.argsort(ids)
        out += [cell[o], off[:, o], u[:, o]]
    recs = eng.diag()
    out.append(np.array([[*r["WE"], *r["WB"], *r["Ekin"], *r["P"]] for r in recs]))
    assert eng.stats()["flags"] == 0
    eng.close()
    return out


# 320 tiles; 24 and 8 particles per cell, and a hot beam whose crossers overflow their queue
@pytest.mark.parametrize("ppc,T,ctas", [(12, 0.3, (3, 2, 4)), (4, 0.3, (3,)), (4, 8.0, (3,)), (12, 8.0, (3, 2, 4))])
def test_variants_bitwise_equal_on_large_grids(pic, ppc, T, ctas):
    wl = pi.weibel_load(ndim=2, nx=320, ny=256, ppc=ppc, T_perp_beam=T, T_bg=0.01 * T, nu=0.1, seed=33)
    ref = None
    for tile in SHAPES:
        for c in ctas:
            got = _run(pic, wl, tile, c, 6)
            if ref is None:
                ref = got
                continue
            for a, b in zip(got[:9], ref[:9]):
                np.testing.assert_array_equal(a, b)
            # the field energies are summed by tile: the order depends on its shape
            np.testing.assert_allclose(got[9], ref[9], rtol=1e-12, atol=1e-12 * np.abs(ref[9]).max())
            np.testing.assert_array_equal(got[9][:, 6:], ref[9][:, 6:])


CHILD = r"""
import json, sys
sys.path.insert(0, "tests")
import numpy as np
import pic_inputs as pi
import paper_0808_4078_gb300 as pic
import test_gpu_variants_large as t
res, arrays = {}, {}
for ppc in (4, 12):
    for T in (0.3, 8.0):
        wl = pi.weibel_load(ndim=2, nx=320, ny=256, ppc=ppc, T_perp_beam=T, T_bg=0.01 * T, nu=0.1, seed=34)
        for i, a in enumerate(t._run(pic, wl, (16, 16), 3, 5)):
            arrays[f"{ppc}_{T}_{i}"] = a
res["lib"] = [l.split()[-1] for l in open("/proc/self/maps") if "libpic" in l][:1]
np.savez(sys.argv[1] + ".npz", **arrays)
json.dump(res, open(sys.argv[1] + ".json", "w"))
"""


def test_large_grids_in_the_bounds_checked_build(pic, tmp_path):
    from paper_0808_4078_gb300 import build
    build.build(debug=True)
    got = []
    for debug in ("1", "0"):
        env = dict(os.environ, PIC_DEBUG_BOUNDS=debug, PYTHONPATH=ROOT + os.pathsep + os.environ.get("PYTHONPATH", ""))
        out = str(tmp_path / debug)
        r = subprocess.run([sys.executable, "-c", CHILD, out], env=env, cwd=ROOT, capture_output=True, text=True,
                           timeout=600)
        assert r.returncode == 0, r.stdout + r.stderr
        lib = json.load(open(out + ".json"))["lib"]
        assert lib and os.path.basename(lib[0]) == ("libpic_debug.so" if debug == "1" else "libpic.so")
        got.append(dict(np.load(out + ".npz")))
    assert got[0].keys() == got[1].keys()
    for k in got[0]:
        np.testing.assert_array_equal(got[0][k], got[1][k])
