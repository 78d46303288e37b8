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


def _warp_block_bytes(net, lanes, td, moments, warps):
    """Shared memory of a block of `warps` warps, from the layout of the kernel: tables, moments, trajectories."""
    m, n, nv = net.n_reactions, net.n_species, 0 if td else len(net.stoi_delta)
    off = m * (24 if td else 16) + nv * 8 + moments + (0 if td else (m + 1) * 4)
    off = (off + 127) // 128 * 128
    pad = (m + lanes - 1) // lanes * lanes
    seg = (pad * 36 + n * 4 + 63) // 128 * 128 + 64
    return off + warps * (32 // lanes) * seg


BLOCK_MAX = 226 * 1024


@pytest.mark.parametrize("m,n,points,warps,table", [(64, 3050, 0, 3, False), (64, 3050, 1, 3, True), (60, 3060, 0, 3, False),
                                                    (64, 2300, 1, 4, True), (128, 5600, 0, 4, False),
                                                    (64, 3050, 2, 3, False)])
def test_blocks_of_three_warps(m, n, points, warps, table):
    """Blocks that four warps do not fit in, beside the largest that they do, with a moment table and without
    (a table above 64 KB is left in global memory)."""
    lanes = 8 if m <= 64 else 16
    net = W.random_mass_action(n, m, 43 + m, 0.5)
    tab = points * n * 16 + points * 8
    tab = tab if tab <= 64 * 1024 else 0
    assert (tab > 0) == table
    assert _warp_block_bytes(net, lanes, False, tab, warps) <= BLOCK_MAX
    assert warps == 4 or _warp_block_bytes(net, lanes, False, tab, warps + 1) > BLOCK_MAX
    x0 = np.random.default_rng(n).poisson(15, n).astype(np.int32)
    t_end = 0.5
    kw = dict(seed=6, max_events=60, sample_dt=1.0 if points <= 1 else t_end / (points - 1))
    g = api.simulate(api.Network(net), x0, t_end, 50, grad=True, grid="moments" if points else "none",
                     mapping=L.RT_MAP_WARP, **kw)
    o = oracle.run(net, x0, t_end, 50, want_grad=True, want_grid=points > 0, n_threads=8, **kw)
    assert_same(g, o, ("x_final", "n_events", "status", "counts", "t_last", "t_internal", "loglik"))
    if points:
        grid = o["grid"].astype(np.int64)
        known = (grid >= 0).all(axis=2)
        assert grid.shape[1] == points
        assert np.array_equal(g["grid_sum"].cpu().numpy(), np.where(known[..., None], grid, 0).sum(0))
        assert np.array_equal(g["grid_sumsq"].cpu().numpy(), np.where(known[..., None], grid * grid, 0).sum(0))
        assert np.array_equal(g["grid_count"].cpu().numpy(), known.sum(0))


def test_moment_table_dropped_where_the_net_changes_fill_the_block():
    """Reactions that make some of every species: with their net changes in shared memory a moment table that would
    do by itself leaves no room for one warp, and the moments are added in global memory."""
    m, n, points = 64, 320, 12
    base = W.random_mass_action(n, m, 5, 0.5)
    rng = np.random.default_rng(8)
    net = W.Network(n, m, base.reac_rxn, base.reac_sp, base.reac_coef, np.repeat(np.arange(m), n),
                    np.tile(np.arange(n), m), rng.integers(1, 3, n * m), base.c)
    tab = points * n * 16 + points * 8
    assert tab <= 64 * 1024 and _warp_block_bytes(net, 8, False, tab, 1) > BLOCK_MAX
    assert _warp_block_bytes(net, 8, False, 0, 4) <= BLOCK_MAX
    x0 = np.full(n, 200, np.int32)
    kw = dict(seed=6, max_events=60, sample_dt=1e-6)
    g = api.simulate(api.Network(net), x0, 1.1e-5, 70, grad=True, grid="moments", mapping=L.RT_MAP_WARP, **kw)
    o = oracle.run(net, x0, 1.1e-5, 70, want_grad=True, want_grid=True, n_threads=8, **kw)
    assert o["n_events"].max() > 5 and o["grid"].shape[1] == points
    assert_same(g, o, ("x_final", "n_events", "status", "counts", "t_last", "t_internal", "loglik"))
    grid = o["grid"].astype(np.int64)
    known = (grid >= 0).all(axis=2)
    assert np.array_equal(g["grid_sum"].cpu().numpy(), np.where(known[..., None], grid, 0).sum(0))
    assert np.array_equal(g["grid_sumsq"].cpu().numpy(), np.where(known[..., None], grid * grid, 0).sum(0))
    assert np.array_equal(g["grid_count"].cpu().numpy(), known.sum(0))
