"""Small networks by the number of trajectories: a warp per trajectory for few (a lane per channel), one
thread per trajectory with its state in shared memory for many (5 to 16 reactions).  Both against the
oracle, and against each other on either side of the sizes where the choice and its variants change.
Every comparison is exact: all define the same bits."""
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

KEYS = ("x_final", "n_events", "status", "counts", "grid", "trace_mu", "trace_t", "t_last", "t_internal", "loglik")


def bits(a):
    return a.view(np.int64) if a.dtype == np.float64 else a


def same(g, o, keys=KEYS):
    for k in keys:
        if k in g and k in o:
            a, b = g[k], o[k]
            a = a.cpu().numpy() if torch.is_tensor(a) else a
            b = b.cpu().numpy() if torch.is_tensor(b) else b.astype(a.dtype)
            assert ((bits(a) == bits(b)) | ((a != a) & (b != b))).all(), k


def net_of(m, n):
    return W.birth_death() if m == 2 and n == 1 else W.random_mass_action(n, m, 70 + 31 * m + n, 0.5)


@pytest.mark.parametrize("mapping", [None, L.RT_MAP_THREAD])
@pytest.mark.parametrize("m,n", [(1, 1), (2, 1), (3, 5), (4, 4), (5, 3), (8, 32), (9, 33), (12, 6), (16, 1), (16, 32)])
def test_against_the_oracle(m, n, mapping):
    net = net_of(m, n)
    x0 = np.full(n, 60, np.int32)
    x0[-1] = 0
    kw = dict(seed=11, stream_id=3, traj_offset=5, sample_dt=0.03, max_events=333)
    for t_end, n_traj in ((0.4, 7), (50.0, 3)):
        g = api.simulate(api.Network(net), x0, t_end, n_traj, grid="traj", grad=True, trace_len=100, mapping=mapping, **kw)
        o = oracle.run(net, x0, t_end, n_traj, want_grid=True, want_grad=True, trace_len=100, n_threads=4, **kw)
        same(g, o)


@pytest.mark.parametrize("m,n,n_traj", [(3, 2, 608), (3, 2, 609), (3, 2, 1216), (3, 2, 1217), (3, 2, 3648), (3, 2, 3649),
                                        (12, 6, 1217), (12, 6, 10944), (12, 6, 10945)])
def test_choice_does_not_change_results(m, n, n_traj):
    net = net_of(m, n)
    x0 = np.random.default_rng(2).integers(0, 90, (n_traj, n)).astype(np.int32)
    x0[n_traj // 2, 0] = -1
    kw = dict(seed=4, sample_dt=0.05, max_events=60, grad=True)
    a = api.simulate(api.Network(net), x0, 0.5, n_traj, grid="moments", **kw)
    b = api.simulate(api.Network(net), x0, 0.5, n_traj, grid="moments", mapping=L.RT_MAP_THREAD, block_threads=64, **kw)
    same(a, b, KEYS + ("grid_sum", "grid_sumsq", "grid_count"))


@pytest.mark.parametrize("n_traj", [9728, 9729])
def test_choice_at_five_reactions(n_traj):
    net = net_of(5, 4)
    x0 = np.random.default_rng(3).integers(0, 90, (n_traj, 4)).astype(np.int32)
    kw = dict(seed=4, max_events=60, grad=True)
    same(api.simulate(api.Network(net), x0, 0.5, n_traj, **kw),
         api.simulate(api.Network(net), x0, 0.5, n_traj, mapping=L.RT_MAP_THREAD, **kw), KEYS)


@pytest.mark.parametrize("n_traj", [3, 20000])
def test_forbidden_channels_overflow_and_absorption(n_traj):
    spec = W.Network(3, 6, [1, 2, 3, 4, 5], [0, 1, 0, 2, 2], [1, 1, 2, 1, 1], [0, 1, 1, 3, 5], [0, 0, 1, 2, 2],
                     [1 << 30, -1, 1, 1, -1], [1.0, 0.5, 2.0, 1e-9, 1.0, 0.3])
    for enabled, x0 in ((None, [5, 5, 2]), ([0, 1, 1, 1, 1, 1], [5, 0, 2]), ([0, 1, 0, 0, 0, 1], [4, 0, 3])):
        net = api.Network(spec).set_enabled(enabled)
        x = np.array(x0, np.int32)
        g = api.simulate(net, x, 30.0, n_traj, seed=9, max_events=500, grad=True)
        o = oracle.run(spec, x, 30.0, 3, seed=9, max_events=500, want_grad=True, enabled=enabled, n_threads=4)
        same({k: v[:3] for k, v in g.items() if k in o}, o)


def test_many_species_still_fit():
    """Enough species that the channel state needs a smaller block."""
    net = net_of(16, 380)
    x0 = np.full(380, 3, np.int32)
    g = api.simulate(api.Network(net), x0, 2.0, 40, seed=2, grad=True, mapping=L.RT_MAP_THREAD)
    same(g, oracle.run(net, x0, 2.0, 40, seed=2, want_grad=True, n_threads=4))
