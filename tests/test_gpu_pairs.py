"""The kernels that work on pairs of cells with packed FP32 arithmetic: bitwise the plain engine's
states and samples (every packed operation is the scalar one in both halves)."""
import numpy as np
import pytest

from workloads import MAGNETITE as M

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def pkg():
    from paper_1912_00310_gb300 import build
    build.build()
    import paper_1912_00310_gb300 as P
    assert torch.cuda.is_available()
    return P


def ensemble(pkg, dims, n_real, *, b=1, dt=2e-15, disp=0.0, shape=0, rate=10000.0, sample_dH=1.0, steps=(113, 37), tune=(),
             plain=False, seed=5):
    """State and samples after `steps` (one advance each) from +z."""
    g = pkg.Grid(*dims, a0=M["a0"], b=b)
    g.set_material(A0=M["A0"], Ms=M["Ms"], K0=M["K0"], alpha=M["alpha"], T=M["T"])
    g.set_scaling(mode=1, Tc=M["Tc"])
    g.set_sweep(H_start=1500.0, H_turn=-1500.0, rate=rate, dt=dt, sample_dH=sample_dH, shape=shape)
    g.set_axis_dispersion(disp)
    g.set_engine(pkg.ENGINE_PLAIN if plain else pkg.ENGINE_RESIDENT)
    for key, value in tune:
        g.set_tuning(key, value)
    g.reset(seed=seed, n_real=n_real, real_offset=11)
    S = torch.zeros((n_real, g.n_samples), device="cuda")
    for k in steps:
        g.advance(k, S)
    m = torch.empty((n_real, g.ncells, 3), device="cuda")
    g.get_state(m)
    g.sync(120.0)
    taken = S[:, 1:sum(steps) // g.sample_every + 1].clone()
    g.close()
    return m, taken


@pytest.mark.parametrize("dims", [(8, 24, 56), (8, 40, 30), (8, 3, 5), (8, 7, 64)])
@pytest.mark.parametrize("disp,shape", [(0.0, 0), (0.0, 1), (0.3, 0), (0.3, 1)])
def test_eight_wide_rods_equal_plain_engine(pkg, dims, disp, shape):
    """Rods eight cells wide, the b = 1 rod and others, with every number of rows per thread that
    holds them (a last row slot that some threads do not use included), both sweeps, with and without
    dispersed axes."""
    ref, ref_s = ensemble(pkg, dims, 3, disp=disp, shape=shape, plain=True)
    assert ref_s.shape[1] >= 3 and torch.isfinite(ref_s).all()
    ran = 0
    for rows in (0, 1, 2, 3, 4):
        try:
            m, s = ensemble(pkg, dims, 3, disp=disp, shape=shape,
                            tune=((pkg.TUNE_ROD_KIND, 2), (pkg.TUNE_ROWS_PER_THREAD, rows)))
        except pkg.LLGError as e:
            assert e.status == 6 and rows == 1  # too many rows for one per thread
            continue
        assert torch.equal(m, ref) and torch.equal(s, ref_s), rows
        ran += 1
    assert ran >= 4


@pytest.mark.parametrize("dims", [(1, 1, 1), (1, 1, 2), (1, 1, 9), (3, 1, 4), (4, 3, 1), (2, 2, 2), (1, 3, 7), (2, 6, 14),
                                  (5, 11, 23), (7, 5, 6), (3, 2, 65), (9, 16, 20), (16, 21, 9)])
@pytest.mark.parametrize("disp,shape", [(0.0, 0), (0.3, 1)])
def test_two_phase_rods_equal_plain_engine(pkg, dims, disp, shape):
    """The two-phase kernel on pairs across the rod's halves: even and odd nz (a last line without its
    upper cells), flat and thin grids (the pair axis moves to y or x), the single cell, one and several
    rods per CTA with a partial last CTA, one, two and four pairs per thread."""
    n_real = 1 if np.prod(dims) > 2000 else 5
    ref, ref_s = ensemble(pkg, dims, n_real, disp=disp, shape=shape, plain=True)
    for rods in (0, 3):
        try:
            m, s = ensemble(pkg, dims, n_real, disp=disp, shape=shape,
                            tune=((pkg.TUNE_ROD_KIND, 1), (pkg.TUNE_RODS_PER_CTA, rods)))
        except pkg.LLGError as e:
            assert e.status == 6 and rods == 3 and np.prod(dims) > 256  # three do not fit a CTA
            continue
        assert torch.equal(m, ref) and torch.equal(s, ref_s), rods


@pytest.mark.parametrize("b,dims,dt", [(2, (4, 12, 28), 5e-15), (4, (2, 6, 14), 10e-15), (8, (1, 3, 7), 20e-15)])
@pytest.mark.parametrize("disp,shape", [(0.0, 0), (0.3, 1)])
def test_row_kernels_equal_plain_engine(pkg, b, dims, dt, disp, shape):
    """The b = 2, 4, 8 rods: one and several rods per CTA, the last CTA partly filled; more steps than
    the 32 whose fields a warp evaluates at once, and a sweep that turns within them."""
    per_step = 1e7 * 1e9 * dt  # Oe: loops of 120, 60 and 30 steps
    kw = dict(b=b, dt=dt, disp=disp, shape=shape, rate=1e7, sample_dH=5 * per_step)
    ref, ref_s = ensemble(pkg, dims, 8, plain=True, **kw)
    for rods in (0, 1, 3):
        try:
            m, s = ensemble(pkg, dims, 8, tune=((pkg.TUNE_ROD_KIND, 3), (pkg.TUNE_RODS_PER_CTA, rods)), **kw)
        except pkg.LLGError as e:
            assert e.status == 6 and rods == 3 and b == 2
            continue
        assert torch.equal(m, ref) and torch.equal(s, ref_s), rods


@pytest.mark.parametrize("dims,n_real", [((8, 24, 56), 2), ((8, 24, 56), 20), ((8, 24, 56), 40), ((4, 12, 28), 3),
                                         ((4, 12, 28), 70), ((5, 11, 23), 3), ((7, 9, 13), 2), ((6, 16, 30), 3),
                                         ((6, 16, 30), 30), ((1, 15, 40), 2), ((3, 30, 20), 2), ((8, 5, 40), 1)])
@pytest.mark.parametrize("disp,shape", [(0.0, 0), (0.3, 1)])
def test_rods_cut_over_several_ctas_equal_plain_engine(pkg, dims, n_real, disp, shape):
    """Few rods: the automatic plan cuts each along z over a cluster of CTAs (2 to 8, even and uneven
    slabs, odd widths, one to four pairs per thread, more clusters than run at once).  Samples after every
    step (the snapshots' double buffer and the partial sums' way through the slabs) and every fifth."""
    for rate, sample_dH, steps in ((1e5, 0.2, (1, 41, 30)), (1e5, 1.0, (113, 37))):
        kw = dict(disp=disp, shape=shape, rate=rate, sample_dH=sample_dH, steps=steps)
        ref, ref_s = ensemble(pkg, dims, n_real, plain=True, **kw)
        m, s = ensemble(pkg, dims, n_real, **kw)
        assert torch.equal(m, ref) and torch.equal(s, ref_s)


@pytest.mark.parametrize("n_real", [1, 7, 1600])
@pytest.mark.parametrize("disp,shape", [(0.0, 0), (0.3, 1)])
def test_small_rods_alone_and_several_to_a_cta_equal_plain_engine(pkg, n_real, disp, shape):
    """The b = 8 rod: one warp each while there are few, three to a CTA (the last one partly filled)
    beyond; samples after every step and past a turn of the sweep."""
    per_step = 1e7 * 1e9 * 20e-15  # Oe: a loop of 30 steps
    kw = dict(b=8, dt=20e-15, disp=disp, shape=shape, rate=1e7, sample_dH=per_step, steps=(1, 33, 14))
    ref, ref_s = ensemble(pkg, (1, 3, 7), n_real, plain=True, **kw)
    m, s = ensemble(pkg, (1, 3, 7), n_real, **kw)
    assert torch.equal(m, ref) and torch.equal(s, ref_s)


@pytest.mark.parametrize("dims", [(7, 12, 20), (9, 13, 26), (12, 12, 21), (8, 16, 20), (2, 31, 26)])
@pytest.mark.parametrize("request_", [(), ("TUNE_RODS_PER_CTA", 3), ("TUNE_ROWS_PER_THREAD", 3), ("TUNE_CELLS_PER_THREAD", 4)])
def test_automatic_plan_of_larger_rods_equals_plain_engine(pkg, dims, request_):
    """Rods of one to four pairs a thread under the automatic plan (200 of them, so that none is cut over
    several CTAs), also where the caller asks for a launch shape and leaves the kernel open."""
    ref, ref_s = ensemble(pkg, dims, 200, disp=0.3, shape=1, steps=(23,), plain=True)
    m, s = ensemble(pkg, dims, 200, disp=0.3, shape=1, steps=(23,),
                    tune=((getattr(pkg, request_[0]), request_[1]),) if request_ else ())
    assert torch.equal(m, ref) and torch.equal(s, ref_s)


@pytest.mark.parametrize("dims,n_real", [((1, 1, 2), 3), ((1, 2, 16), 200), ((3, 11, 1), 3), ((4, 8, 4), 3), ((3, 43, 1), 3), ((2, 4, 20), 200), ((7, 23, 1), 3),
                                         ((3, 4, 26), 152), ((3, 4, 26), 153), ((4, 10, 10), 40)])
@pytest.mark.parametrize("disp,shape", [(0.0, 0), (0.3, 1)])
def test_small_rods_a_cell_to_a_thread_equal_plain_engine(pkg, dims, n_real, disp, shape):
    """Rods of one warp (2 and 32 cells), a cell more (33), of four warps and a cell more (128, 129), and up to the sizes and ensembles at which the
    pair kernel takes over (160 and 161 cells; 312 cells with as many rods as SMs and one more; 400)."""
    kw = dict(disp=disp, shape=shape, steps=(1, 50, 23), sample_dH=0.2, rate=1e5)
    ref, ref_s = ensemble(pkg, dims, n_real, plain=True, **kw)
    m, s = ensemble(pkg, dims, n_real, tune=((pkg.TUNE_ROD_KIND, 1),), **kw)
    assert torch.equal(m, ref) and torch.equal(s, ref_s)
    m, s = ensemble(pkg, dims, n_real, **kw)
    assert torch.equal(m, ref) and torch.equal(s, ref_s)


@pytest.mark.parametrize("n_real", [150, 400])
@pytest.mark.parametrize("disp,shape", [(0.0, 0), (0.3, 1)])
def test_row_kernel_with_one_and_two_ctas_to_an_sm_equals_plain_engine(pkg, n_real, disp, shape):
    """The b = 2 rod with at most one rod to an SM and with more."""
    kw = dict(b=2, dt=5e-15, disp=disp, shape=shape, steps=(41,))
    ref, ref_s = ensemble(pkg, (4, 12, 28), n_real, plain=True, **kw)
    m, s = ensemble(pkg, (4, 12, 28), n_real, tune=((pkg.TUNE_ROD_KIND, 3),), **kw)
    assert torch.equal(m, ref) and torch.equal(s, ref_s)
