"""The block routine by slots per thread (1 to 8, exact or with entries past M), by the number of
trajectories that sets its block size, with so many species that the channel state stays out of shared
memory, and in a batch beside the other classes.  All comparisons are exact."""
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


@pytest.mark.parametrize("m,n,b", [(1, 1, 64), (33, 7, 32), (64, 9, 64), (257, 40, 0), (511, 60, 64), (512, 60, 64),
                                   (513, 60, 128), (600, 4, 96), (1025, 200, 0), (2047, 300, 512), (2049, 300, 512),
                                   (2049, 300, 288), (3000, 90, 416), (3585, 700, 512), (4096, 1024, 512),
                                   (300, 36000, 0), (2000, 42000, 256)])
def test_slots(m, n, b):
    net = W.pure_birth() if m == 1 else W.random_mass_action(n, m, 500 + m + b, 0.7)
    x0 = np.random.default_rng(m).poisson(20, net.n_species).astype(np.int32)
    kw = dict(seed=3, max_events=150, sample_dt=0.001)
    g = api.simulate(api.Network(net), x0, 0.05, 4, grad=True, grid="traj" if n < 2000 else "none", trace_len=50,
                     mapping=L.RT_MAP_BLOCK, block_threads=b, **kw)
    o = oracle.run(net, x0, 0.05, 4, want_grad=True, want_grid=n < 2000, trace_len=50, n_threads=4, **kw)
    assert_same(g, o, ("x_final", "n_events", "status", "counts", "grid", "t_last", "t_internal", "loglik",
                       "trace_mu", "trace_t"))


@pytest.mark.parametrize("n_traj", [1, 153, 700, 3000])
def test_block_size_by_trajectories(n_traj):
    net = W.random_mass_action(100, 700, 9, 0.7)
    x0 = np.full(100, 20, np.int32)
    g = api.simulate(api.Network(net), x0, 1.0, n_traj, seed=6, max_events=40, grad=True)
    o = oracle.run(net, x0, 1.0, n_traj, seed=6, max_events=40, want_grad=True, n_threads=8)
    assert_same(g, o)


@pytest.mark.parametrize("block_threads,n_big", [(512, 300), (128, 300), (512, 36000)])
def test_batch_of_every_class(block_threads, n_big):
    sizes = [(1, 1), (3, 2), (8, 9), (20, 5), (200, 40), (256, 64), (257, 60), (512, 100), (513, 100), (1500, n_big),
             (1024, 200), (2000, 100)]
    specs = [W.pure_birth() if m == 1 else W.random_mass_action(n, m, 60 + m, 0.6) for m, n in sizes]
    x0s = [np.full(s.n_species, 15, np.int32) for s in specs]
    batch = api.Batch(specs, block_threads=block_threads)
    nt = 3
    out = batch.run(torch.from_numpy(np.concatenate(x0s)).cuda(), torch.full((len(specs),), 0.4, dtype=torch.float64).cuda(),
                    nt, seed=7, max_events=120, outputs=batch.outputs(nt, grad=True))
    for i, s in enumerate(specs):
        o = oracle.run(s, x0s[i], 0.4, nt, seed=7, stream_id=i, max_events=120, want_grad=True, n_threads=4)
        g = dict(x_final=batch.x_final_of(out, i, nt), n_events=out["n_events"][i], status=out["status"][i],
                 t_last=out["t_last"][i], loglik=out["loglik"][i], counts=batch.per_channel_of(out, "counts", i, nt),
                 t_internal=batch.per_channel_of(out, "t_internal", i, nt))
        assert_same(g, o)


@pytest.mark.parametrize("n_traj", [1, 153, 1300])
def test_species_limit_does_not_depend_on_the_trajectories(n_traj):
    """The most species that the smallest block (64 threads here) is given run with every number of
    trajectories, one more is refused with every number."""
    m, b = 300, 64
    n = (200 * 1024 - m * 4 - (m + 31) // 32 * 4 - b // 32 * 24 - b * 8 - 96) // 4
    net = W.random_mass_action(n, m, 71, 0.7)
    x0 = np.random.default_rng(2).poisson(20, n).astype(np.int32)
    kw = dict(seed=4, max_events=40)
    g = api.simulate(api.Network(net), x0, 1.0, n_traj, grad=True, **kw)
    few = min(n_traj, 3)
    o = oracle.run(net, x0, 1.0, few, want_grad=True, n_threads=4, **kw)
    assert_same({k: v[:few] for k, v in g.items() if not k.startswith("_")}, o)
    wide = W.random_mass_action(n + 1, m, 71, 0.7)
    with pytest.raises(L.RandtimeError):
        api.simulate(api.Network(wide), np.zeros(n + 1, np.int32), 1.0, n_traj, **kw)


@pytest.mark.parametrize("m,tiny", [(600, 6), (600, 7), (600, 8), (600, 9), (600, 31), (600, 33), (600, 599), (2000, 1500),
                                    (300, 40)])
@pytest.mark.parametrize("rate", [1e-45, 1e-320, 1e40])
def test_many_candidates(m, tiny, rate):
    """Channels whose rates no float bound covers are candidates of every event: lists of a few, of more than a
    warp, and of every channel."""
    n = m // 4
    net = W.random_mass_action(n, m, 81, 0.7)
    c = net.c.copy()
    if rate > 1:
        c *= rate
    c[np.random.default_rng(m + tiny).permutation(m)[:tiny]] = rate
    x0 = np.random.default_rng(m).poisson(60, n).astype(np.int32)
    t_end = 1e-30 if rate > 1 else 1e6
    kw = dict(seed=11, max_events=120)
    for n_traj in (2, 700 if m == 300 else 3):  # a block of one slot per thread, and of several
        g = api.simulate(api.Network(net.with_rates(c)), x0, t_end, n_traj, grad=True, mapping=L.RT_MAP_BLOCK, **kw)
        o = oracle.run(net.with_rates(c), x0, t_end, n_traj, want_grad=True, n_threads=8, **kw)
        assert_same(g, o)
