"""Rods cut over several CTAs: the waits' limit."""
import pytest

from test_gpu_pairs import ensemble, pkg  # noqa: F401  (pkg: the fixture)

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
