"""Field energies of the diagnostic record on grids of more than 1024 tiles, whose partials are summed
in pieces of 256 tiles: against numpy's FP64 sums of the same fields (FP64 rounding of the order of
the sums: 1e-12), and the same bits alone and in a batch whose other runs shift its tiles."""
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


# 1024, 1025, 1280, 1281, 2600 tiles in 2D; 1024, 1027, 1300 in 3D
@pytest.mark.parametrize("shape", [(512, 512), (16, 16 * 1025), (16, 16 * 1280), (16, 16 * 1281), (400, 1664),
                                   (64, 64, 64), (8, 8, 4 * 1027), (80, 104, 40)])
def test_field_energies(pic, shape):
    nd, n = len(shape), int(np.prod(shape))
    nz = shape[2] if nd == 3 else 1
    eng = pic.Engine(nd, shape[0], shape[1], nz, dx=0.1, dt=0.05, capacity=(64, 64), diag_interval=1)
    rng = np.random.default_rng(n)
    E0, B0 = rng.standard_normal((2, 3, n)).astype(np.float32)
    eng.set_fields(E0, B0)
    want = [(E0, B0)]
    for _ in range(2):
        eng.step(1)
        want.append(eng.fields()[:2])
    recs = eng.diag()
    eng.close()
    assert len(recs) == 2
    for rec, (E, B) in zip(recs, want):
        for got, F in ((rec["WE"], E), (rec["WB"], B)):
            w = (F.astype(np.float64) ** 2).sum(axis=1) * 0.1 ** nd
            np.testing.assert_allclose(got, w, rtol=1e-12)


@pytest.mark.parametrize("ndim", [2, 3])
def test_long_run_in_a_batch(pic, ndim):
    grid = dict(nx=16, ny=16 * 1030) if ndim == 2 else dict(nx=8, ny=8, nz=4 * 1030)
    small = dict(nx=32, ny=48) if ndim == 2 else dict(nx=16, ny=8, nz=12)
    long = pi.weibel_load(ndim=ndim, ppc=1, T_perp_beam=0.2, T_bg=0.01, seed=3, **grid)
    short = pi.weibel_load(ndim=ndim, ppc=2, T_perp_beam=0.2, T_bg=0.01, seed=4, **small)
    kw = dict(diag_interval=1, diag_capacity=16)
    alone = [pic.Engine.from_workloads([w], **kw) for w in (short, long)]
    batch = pic.Engine.from_workloads([short, long, short, long], **kw)
    for eng in (*alone, batch):
        eng.step(9)
    for r in range(4):
        a, b = alone[r % 2].diag(run=0), batch.diag(run=r)
        assert len(a) == len(b) == 9
        for x, y in zip(a, b):
            for k in x:
                np.testing.assert_array_equal(np.asarray(x[k]), np.asarray(y[k]))
    for eng in (*alone, batch):
        eng.close()
