"""Rods cut over several CTAs: the waits' limit and what happens when one runs out."""
import math

import numpy as np
import pytest

from test_cut_plan import CASES
from test_gpu_pairs import ensemble, pkg  # noqa: F401  (pkg: the fixture)
from workloads import MAGNETITE as M

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("dims,n_real,b,dt", [((4, 12, 28), 3, 2, 5e-15), ((8, 24, 56), 2, 1, 2e-15)])
def test_samples_further_apart_than_the_wait_limit(pkg, dims, n_real, b, dt):  # noqa: F811
    """The limit of a cut rod's waits holds for its neighbours' lines, not for the steps between two samples:
    samples 20000 steps apart (tens of milliseconds) under a limit of 2 ms are the plain engine's, and no
    wait gives up (ensemble() synchronises and would raise)."""
    every = 20000
    per_step = 1000.0 * 1e9 * dt  # Oe
    kw = dict(b=b, dt=dt, rate=1000.0, sample_dH=every * per_step, steps=(every + 7, every + 1))
    ref, ref_s = ensemble(pkg, dims, n_real, plain=True, **kw)
    assert ref_s.shape[1] == 2
    m, s = ensemble(pkg, dims, n_real, tune=((pkg.TUNE_HANDOFF_TIMEOUT_MS, 2),), **kw)
    assert torch.equal(m, ref) and torch.equal(s, ref_s)


def test_samples_seconds_apart(pkg):  # noqa: F811
    """The same under the default limit, 750000 steps (2.6 s) to the sample within one launch."""
    kw = dict(rate=1000.0, sample_dH=1500.0, steps=(750_007,))
    ref, ref_s = ensemble(pkg, (8, 24, 56), 32, tune=((pkg.TUNE_ROD_KIND, 2),), **kw)
    assert ref_s.shape[1] == 1
    m, s = ensemble(pkg, (8, 24, 56), 32, **kw)
    assert torch.equal(m, ref) and torch.equal(s, ref_s)


def cut_grid(pkg, dims):  # noqa: F811
    g = pkg.Grid(*dims, a0=M["a0"])
    g.set_material(A0=M["A0"], Ms=M["Ms"], K0=M["K0"], alpha=M["alpha"], T=M["T"])
    g.set_scaling(mode=1, Tc=M["Tc"])
    g.set_sweep(H_start=1500.0, H_turn=-1500.0, rate=1e5, dt=2e-15, sample_dH=0.2)  # a sample every step
    g.set_engine(pkg.ENGINE_RESIDENT)
    return g


@pytest.mark.parametrize("dims,n_real", [c[0:3:2] for c in CASES])
def test_wait_that_runs_out_then_recovery(pkg, dims, n_real):  # noqa: F811
    """With the lines to the slab below withheld on purpose and a limit of 20 ms every rod's CTAs give up: the
    launch ends, llg_sync reports ETIMEOUT (which shows that the rods were cut: no other kernel waits with fewer
    rods than SMs), no sample is written and the state stays what it was.  The same context then runs
    normally, bitwise the plain engine."""
    g = cut_grid(pkg, dims)
    g.set_tuning(pkg.TUNE_HANDOFF_TIMEOUT_MS, 20)
    g.set_tuning(pkg.TUNE_WITHHOLD_HANDOFF, 1)
    g.reset(seed=3, n_real=n_real)
    before = torch.empty((n_real, g.ncells, 3), device="cuda")
    g.get_state(before)
    S = torch.full((n_real, g.n_samples), 7.0, device="cuda")
    g.advance(50, S)
    with pytest.raises(pkg.LLGError) as e:
        g.sync(120)
    assert e.value.status == 5 and "hand-off" in str(e.value)
    after = torch.empty_like(before)
    g.get_state(after)
    assert torch.equal(after, before) and bool((S == 7.0).all())
    g.set_tuning(pkg.TUNE_WITHHOLD_HANDOFF, 0)
    out = []
    for engine in (pkg.ENGINE_RESIDENT, pkg.ENGINE_PLAIN):
        g.set_engine(engine)
        g.reset(seed=3, n_real=n_real)
        S.fill_(7.0)
        g.advance(50, S)
        g.get_state(after)
        g.sync(120)
        out.append((after.clone(), S.clone()))
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
    g.close()


def test_gradient_reports_a_wait_that_ran_out(pkg):  # noqa: F811
    """The gradient's forward pass may cut its rods too: a wait that runs out there is ETIMEOUT and no loss, the
    ensemble (whose state the gradient does not touch) is not marked, and the next gradient is the one that
    the rods give uncut."""
    g = cut_grid(pkg, (5, 11, 17))  # 935 cells
    g.reset(seed=3, n_real=3)
    target = np.linspace(1.0, -1.0, g.n_samples)
    g.set_tuning(pkg.TUNE_HANDOFF_TIMEOUT_MS, 20)
    g.set_tuning(pkg.TUNE_WITHHOLD_HANDOFF, 1)
    with pytest.raises(pkg.LLGError) as e:
        g.loss_grad(100, target, 0, 64)
    assert e.value.status == 5 and "hand-off" in str(e.value)
    g.sync(60)
    g.set_tuning(pkg.TUNE_WITHHOLD_HANDOFF, 0)
    L, grad = g.loss_grad(100, target, 0, 64)
    g.set_tuning(pkg.TUNE_BALANCE, 0)  # one SM a rod
    L1, grad1 = g.loss_grad(100, target, 0, 64)
    assert L == L1 and np.array_equal(grad, grad1)
    g.close()


@pytest.mark.parametrize("n_real", [3, 200])
def test_gradient_of_a_non_finite_state(pkg, n_real):  # noqa: F811
    """A loss that is not a number is returned as such and reported by the next llg_sync."""
    g = cut_grid(pkg, (5, 11, 17))
    g.reset(seed=3, n_real=n_real)
    m = torch.zeros((n_real, g.ncells, 3), device="cuda")
    m[..., 2] = 1.0
    m[1, 7, 0] = float("nan")
    g.set_state(m, 0)
    L, _ = g.loss_grad(100, np.zeros(g.n_samples), 0, 64)
    assert math.isnan(L)
    with pytest.raises(pkg.LLGError) as e:
        g.sync(60)
    assert e.value.status == 4
    g.close()


def test_rods_stay_whole_beside_other_streams(pkg):  # noqa: F811
    """A context on a stream of its own may run beside others, which a cut rod would take SMs from: its rods are
    not cut (no wait to run out), the context moved to the default stream cuts them; the states agree."""
    g = cut_grid(pkg, (4, 12, 28))
    g.set_tuning(pkg.TUNE_HANDOFF_TIMEOUT_MS, 20)
    g.set_tuning(pkg.TUNE_WITHHOLD_HANDOFF, 1)
    out = []
    stream = torch.cuda.Stream()
    for own in (True, False):
        g.set_stream(stream.cuda_stream if own else 0)
        g.reset(seed=3, n_real=3)
        g.advance(50)
        if own:
            g.sync(60)
        else:
            with pytest.raises(pkg.LLGError) as e:
                g.sync(60)
            assert e.value.status == 5
            g.set_tuning(pkg.TUNE_WITHHOLD_HANDOFF, 0)
            g.reset(seed=3, n_real=3)
            g.advance(50)
            g.sync(60)
        m = torch.empty((3, g.ncells, 3), device="cuda")
        g.get_state(m)
        g.sync(60)
        out.append(m.clone())
    torch.cuda.synchronize()
    assert torch.equal(out[0], out[1])
    g.close()
