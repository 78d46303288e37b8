"""What the library chooses by itself is not slower than what a caller can name: the same call timed both ways on
the device, the shorter of several runs of each.  The lines of these choices were measured; a tenth is allowed."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2103_00405_gb300 import workloads as W

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - CPU-only hosts skip the GPU suite
    pytest.skip("CUDA not available", allow_module_level=True)

from paper_2103_00405_gb300 import _lib as L  # noqa: E402
from paper_2103_00405_gb300 import api  # noqa: E402


def ms(fn, runs=7):
    fn()
    best = float("inf")
    for _ in range(runs):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        fn()
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b))
    return best


@pytest.mark.parametrize("n_traj", [20, 600, 1800])
@pytest.mark.parametrize("m", [17, 32, 64, 100])
def test_ramped_segment_width_by_trajectories(m, n_traj):
    n = max(4, m // 4)
    net = api.Network(W.random_mass_action(n, m, W.GEN_SEED_BASE + m, 0.5))
    rng = np.random.default_rng(m)
    net.set_rate_slopes(np.where(rng.random(m) < 0.3, 0.0, rng.uniform(0.1, 3.0, m)))
    x0 = torch.from_numpy(rng.poisson(100, n).astype(np.int32)).cuda()
    out = {}

    def run(lanes):
        return lambda: api.simulate(net, x0, 1.0, n_traj, seed=7, max_events=500, lanes_per_traj=lanes, outputs=out)

    assert ms(run(0)) <= 1.1 * ms(run(32))


@pytest.mark.parametrize("m,n_traj", [(3, 152 * 23), (5, 152 * 40), (5, 152 * 70), (8, 152 * 71), (12, 152 * 71)])
def test_few_trajectories_of_a_small_network(m, n_traj):
    n = 6
    net = api.Network(W.random_mass_action(n, m, W.GEN_SEED_BASE + m, 0.5))
    x0 = torch.from_numpy(np.random.default_rng(m).poisson(200, n).astype(np.int32)).cuda()
    out = {}

    def run(mapping):
        return lambda: api.simulate(net, x0, 2.0, n_traj, seed=7, max_events=600, mapping=mapping, outputs=out)

    assert ms(run(None)) <= 1.1 * ms(run(L.RT_MAP_THREAD))


def test_rates_that_no_float_bound_covers():
    """A third of the channels with rates of 1e-45: every one is computed exactly at every event, which may cost
    as much again as the event and half as much more, not several times it."""
    m, n = 3000, 750
    spec = W.random_mass_action(n, m, W.GEN_SEED_BASE + m, 0.5)
    x0 = torch.from_numpy(np.random.default_rng(m).poisson(100, n).astype(np.int32)).cuda()
    out = {}

    def run(rate):
        c = spec.c.copy()
        c[-m // 3:] = rate
        net = api.Network(spec.with_rates(c))
        return lambda: api.simulate(net, x0, 1e6, 64, seed=7, max_events=500, outputs=out)

    assert ms(run(1e-45)) <= 2.5 * ms(run(1e-12))


@pytest.mark.parametrize("m", [64, 128, 200, 256])
def test_runs_that_fire_no_event(m):
    """The increments of the next firings are not drawn before one is needed: a run that stops before its first
    event takes at most six tenths of one with ten events."""
    net = api.Network(W.random_mass_action(m // 4, m, W.GEN_SEED_BASE + m, 0.5))
    x0 = torch.from_numpy(np.random.default_rng(m).poisson(100, m // 4).astype(np.int32)).cuda()
    out = {}

    def run(events):
        return lambda: api.simulate(net, x0, 5.0, 100000, seed=7, max_events=events, outputs=out)

    assert ms(run(0)) <= 0.6 * ms(run(10))
