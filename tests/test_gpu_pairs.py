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


def ensemble(pkg, dims, n_real, *, b=1, dt=2e-15, disp=0.0, shape=0, rate=10000.0, steps=(113, 37), tune=(), plain=False,
             seed=5):
    """State and samples after `steps` (one advance each) from +z."""
    g = pkg.Grid(*dims, a0=M["a0"], b=b)
    g.set_material(A0=M["A0"], Ms=M["Ms"], K0=M["K0"], alpha=M["alpha"], T=M["T"])
    g.set_scaling(mode=1, Tc=M["Tc"])
    g.set_sweep(H_start=1500.0, H_turn=-1500.0, rate=rate, dt=dt, sample_dH=1.0, shape=shape)
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
