"""Moment recorder (pic_record_moments) against the oracle's definitions (oracle.closure).

Both sides step the same seeded workload independently (the GPU in FP32, the oracle in FP64)
and record the coarse moments of their own states.  Field seeds of amplitude 0.05 make the
particle forces and the fluctuation friction non-trivial.  Tolerances: the states agree to
~1e-5 relative after a few steps (parity tests), the sums are int64 fixed point 2^-30:
densities 1e-6 relative; means, variances, W_ES and forces 1e-4 of their row's scale; the label
where the return-current drift is not small.
"""
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


def _seed_fields(eng, sim, wl, amp=0.05, seed=9):
    rng = np.random.default_rng(seed)
    E0 = (amp * rng.standard_normal((3, wl.ncell))).astype(np.float32)
    B0 = (amp * rng.standard_normal((3, wl.ncell))).astype(np.float32)
    eng.set_fields(E0, B0)
    shape = sim.E[0].shape
    for a in range(3):
        sim.E[a][...] = E0[a].reshape(shape)
        sim.B[a][...] = B0[a].reshape(shape)


def _compare(got, want):
    for r in range(12):
        g, w = got[r].astype(np.float64), want[r]
        scale = np.abs(w).max() + 1e-12
        if r < 2:
            assert np.allclose(g, w, rtol=1e-6, atol=1e-9), r
        elif r < 11:
            assert np.abs(g - w).max() <= 1e-4 * scale + 1e-7, (r, np.abs(g - w).max(), scale)
    ok = np.abs(want[3]) > 0.5 * np.abs(want[3]).max()
    lab_g, lab_w = got[11].astype(np.float64)[ok], want[11][ok]
    assert np.abs(lab_g - lab_w).max() <= 1e-3 * (np.abs(lab_w).max() + 1e-6)


@pytest.mark.parametrize("ndim", [3, 2])
def test_moments_match_oracle(pic, ndim):
    import oracle
    from oracle import closure
    if ndim == 3:
        wl = pi.weibel_load(ndim=3, nx=16, ny=16, nz=16, ppc=8, T_perp_beam=0.2, T_bg=0.01,
                            nu=0.1, seed=61)
    else:
        wl = pi.weibel_load(ndim=2, nx=32, ny=32, ppc=16, T_perp_beam=0.2, T_bg=0.01, nu=0.1,
                            seed=62)
    eng = pic.Engine.from_workload(wl, track_ids=True)
    sim = oracle.Simulation.from_workload(wl)
    _seed_fields(eng, sim, wl)
    eng.step(3)
    sim.step(3, record=False)
    got = eng.record_moments(4, 4).cpu().numpy()
    want = closure.coarse_moments(sim, 4, 4)
    assert got.shape == want.shape
    _compare(got, want)
    # bitwise reproducible
    again = eng.record_moments(4, 4).cpu().numpy()
    assert np.array_equal(got, again)
    eng.close()


def test_moments_reject_bad_blocks(pic):
    wl = pi.weibel_load(ndim=2, nx=32, ny=32, ppc=4, seed=63)
    eng = pic.Engine.from_workload(wl)
    with pytest.raises(pic.PicError):
        eng.record_moments(5, 4)
    with pytest.raises(pic.PicError):
        eng.record_moments(4, 4, run=1)
    eng.close()


@pytest.mark.parametrize("bx,by,ppc,nu,w_beam", [(1, 1, 3, 0.0, 0.1), (2, 8, 5, 0.1, 0.1), (8, 2, 40, 0.0, 0.1),
                                                (16, 16, 2, 0.0, 0.1), (4, 4, 1, 0.0, 40.0)])
def test_columns_per_tile_of_the_3d_recorder(pic, bx, by, ppc, nu, w_beam):
    """1 to 64 coarse columns per 8 x 8 x 4 tile, few and many particles per tile, and a weight
    whose terms leave the 32-bit words (|w u| 2^36 >= 2^40)."""
    import oracle
    from oracle import closure
    wl = pi.weibel_load(ndim=3, nx=16, ny=32, nz=12, ppc=ppc, T_perp_beam=0.2, T_bg=0.01, nu=nu, seed=21)
    eng = pic.Engine.from_workload(wl, diag_interval=0)
    sim = oracle.Simulation.from_workload(wl)
    if w_beam != 0.1:
        eng.close()
        wl.species[0].w = w_beam
        eng = pic.Engine.from_workload(wl, diag_interval=0)
        sim = oracle.Simulation.from_workload(wl)
    _seed_fields(eng, sim, wl)
    got = eng.record_moments(bx, by).cpu().numpy()
    _compare(got, closure.coarse_moments(sim, bx, by))
    eng.close()


def _crowded(ndim, seed):
    """Particles in the first 3/8 of the cells only, 16 per cell there."""
    import dataclasses
    kw = dict(nz=16) if ndim == 3 else {}
    wl = pi.weibel_load(ndim=ndim, nx=32, ny=32, ppc=16, T_perp_beam=0.5, T_bg=0.05, nu=0.1, seed=seed, **kw)
    full = 32 * 32 * (16 if ndim == 3 else 1) * 3 // 8
    sp = []
    for s in wl.species:
        k = s.cell < full
        sp.append(dataclasses.replace(s, cell=s.cell[k], offset=s.offset[:, k], u=s.u[:, k]))
    return dataclasses.replace(wl, species=sp)


@pytest.mark.parametrize("ndim", [2, 3])
def test_spilled_particles_give_the_same_bits_as_slots(pic, ndim):
    """A record does not depend on which particles are in the spill list (an order of atomics): tight
    slots against room for all, and a rerun, bitwise."""
    wl = _crowded(ndim, 64)
    rng = np.random.default_rng(7)
    E0, B0 = (0.05 * rng.standard_normal((2, 3, wl.ncell))).astype(np.float32)
    got = []
    for cc in ((12, 12), (12, 12), (128, 128)):
        eng = pic.Engine.from_workload(wl, diag_interval=0, sort_interval=8, cell_capacity=cc)
        eng.set_fields(E0, B0)
        eng.step(3)
        spilled = min(eng.stats()["spilled"])
        assert spilled > 0 if cc[0] == 12 else spilled == 0
        got.append(eng.record_moments(4, 4).cpu().numpy())
        eng.close()
    for other in got[1:]:
        np.testing.assert_array_equal(got[0], other)


@pytest.mark.parametrize("nz,scale", [(4, 1.0), (12, 1.0), (64, 1e-3)])
def test_column_sums_are_those_of_fp64(pic, nz, scale):
    """W_ES of single columns (bx = by = 1) of given fields: FP64 sums of FP64 deviations, rounded to
    FP32 once, so within half an FP32 unit in the last place of numpy's (and the FP64 rounding of a few
    dozen terms, far below 1e-6 of that unit).  A deviation rounded to FP32 misses this in a large
    share of the columns."""
    wl = pi.weibel_load(ndim=3, nx=16, ny=16, nz=nz, ppc=1, T_perp_beam=0.1, T_bg=0.01, seed=71)
    eng = pic.Engine.from_workload(wl, diag_interval=0)
    rng = np.random.default_rng(nz)
    E0, B0 = (scale * rng.standard_normal((2, 3, wl.ncell)) + 0.7 * scale).astype(np.float32)
    eng.set_fields(E0, B0)
    got = eng.record_moments(1, 1).cpu().numpy()[8].astype(np.float64)
    eng.close()
    E = E0.astype(np.float64).reshape(3, nz, 256)
    want = ((E - E.mean(axis=1, keepdims=True)) ** 2).sum(axis=0).mean(axis=0)
    ulp = np.spacing(want.astype(np.float32)).astype(np.float64)
    assert (np.abs(got - want) <= 0.5001 * ulp).all()
