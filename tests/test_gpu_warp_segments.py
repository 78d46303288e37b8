"""Warp segments with shared-memory state (constant and time-dependent rates) where their bounds and
layouts can go wrong: channel counts at the edges of the segment widths, slopes and rates far out of the
float range, and so many species or grid points that a block holds fewer warps or no moment table.  All
comparisons are exact."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_2103_00405_gb300 import workloads as W

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - CPU-only hosts skip the GPU suite
    pytest.skip("CUDA not available", allow_module_level=True)

from paper_2103_00405_gb300 import _lib as L  # noqa: E402
from paper_2103_00405_gb300 import api  # noqa: E402

from test_gpu_parity import assert_same  # noqa: E402


@pytest.mark.parametrize("lanes", [0, 32])
@pytest.mark.parametrize("m", [1, 8, 9, 16, 17, 63, 64, 65, 127, 129, 255, 256])
def test_ramped_widths(m, lanes):
    n = max(1, m // 5)
    net = W.pure_birth() if m == 1 else W.random_mass_action(n, m, 300 + m, 0.5)
    n = net.n_species
    rng = np.random.default_rng(m)
    beta = np.where(rng.random(m) < 0.3, 0.0, rng.uniform(0.1, 3.0, m))
    x0 = np.full(n, 30, np.int32)
    kw = dict(seed=5, max_events=120, sample_dt=0.02)
    g = api.simulate(api.Network(net).set_rate_slopes(beta), x0, 0.3, 9, grad=True, grid="traj",
                     mapping=L.RT_MAP_WARP, lanes_per_traj=lanes, **kw)
    o = oracle.run(net, x0, 0.3, 9, beta=beta, want_grad=True, want_grid=True, n_threads=4, **kw)
    assert_same(g, o)


@pytest.mark.parametrize("b", [1e-320, 1e-60, 1e-12, 1e6, 1e25, 1e120])
@pytest.mark.parametrize("scale", [1e-200, 1e-15, 1.0, 1e15, 1e200])
def test_ramped_slopes_and_rates_far_out(b, scale):
    m, n = 30, 8
    net = W.random_mass_action(n, m, 17, 0.5)
    c = net.c.copy()
    c[::2] *= scale
    net = net.with_rates(c)
    beta = np.where(np.arange(m) % 3 == 0, 0.0, np.where(np.arange(m) % 3 == 1, b, 0.7))
    x0 = np.full(n, 25, np.int32)
    g = api.simulate(api.Network(net).set_rate_slopes(beta), x0, 1e4, 5, seed=8, max_events=90, grad=True,
                     mapping=L.RT_MAP_WARP)
    o = oracle.run(net, x0, 1e4, 5, seed=8, max_events=90, beta=beta, want_grad=True, n_threads=4)
    assert_same(g, o)


@pytest.mark.parametrize("m,n,t_end", [(64, 2900, 2.0), (256, 5000, 1.0), (40, 10, 60.0)])
def test_fewer_warps_per_block_and_no_moment_table(m, n, t_end):
    net = W.random_mass_action(n, m, 41 + m, 0.5)
    x0 = np.full(n, 3, np.int32)
    kw = dict(seed=6, max_events=300, sample_dt=0.01)
    a = api.simulate(api.Network(net), x0, t_end, 50, grad=True, grid="moments", mapping=L.RT_MAP_WARP, **kw)
    o = oracle.run(net, x0, t_end, 50, want_grad=True, want_grid=True, n_threads=8, **kw)
    assert_same(a, o, ("x_final", "n_events", "status", "counts", "t_last", "t_internal", "loglik"))
    grid = o["grid"].astype(np.int64)
    known = (grid >= 0).all(axis=2)
    assert np.array_equal(a["grid_sum"].cpu().numpy(), np.where(known[..., None], grid, 0).sum(0))
    assert np.array_equal(a["grid_sumsq"].cpu().numpy(), np.where(known[..., None], grid * grid, 0).sum(0))
    assert np.array_equal(a["grid_count"].cpu().numpy(), known.sum(0))


@pytest.mark.parametrize("m,n,n_traj", [(20, 5, 152 * 12), (20, 5, 152 * 12 + 1), (90, 20, 152 * 12 + 1),
                                        (64, 2700, 1900), (64, 3300, 1900), (20, 12000, 1900), (100, 12000, 30)])
def test_ramped_widths_by_trajectories_and_species(m, n, n_traj):
    """Both sides of the lines between 32 lanes and the width by M: few trajectories, many species."""
    net = W.random_mass_action(n, m, 7 + m, 0.5)
    beta = np.where(np.arange(m) % 3 == 0, 0.0, 0.4)
    x0 = np.random.default_rng(n).poisson(20, n).astype(np.int32)
    kw = dict(seed=9, max_events=40)
    g = api.simulate(api.Network(net).set_rate_slopes(beta), x0, 0.5, n_traj, grad=True, mapping=L.RT_MAP_WARP, **kw)
    o = oracle.run(net, x0, 0.5, n_traj, beta=beta, want_grad=True, n_threads=8, **kw)
    assert_same(g, o)
