"""The bundle kernel's variants: networks whose net changes do not fit the packed dependency records, one
channel firing again and again (its sum of increments is used before memory is read again), slices of every
size, and the range check of a firing.  All comparisons are exact."""
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


def check(net, x0, n_traj=3, max_events=200, **kw):
    run = dict(seed=5, max_events=max_events)
    g = api.simulate(api.Network(net), x0, 1e6, n_traj, grad=True, trace_len=max_events, mapping=L.RT_MAP_BUNDLE, **run,
                     **kw)
    o = oracle.run(net, x0, 1e6, n_traj, want_grad=True, trace_len=max_events, n_threads=4, **run)
    assert_same(g, o, ("x_final", "n_events", "status", "counts", "t_last", "t_internal", "loglik", "trace_mu", "trace_t"))
    return o


@pytest.mark.parametrize("ctas", [1, 3, 40])
def test_records_that_do_not_pack(ctas):
    base = W.random_mass_action(60, 2900, 4, 0.8)
    # reaction 7 also makes six other species, reaction 8 two hundred molecules of one
    rxn = np.concatenate([base.stoi_rxn, np.full(6, 7), [8]])
    sp = np.concatenate([base.stoi_sp, np.arange(40, 46), [50]])
    d = np.concatenate([base.stoi_delta, np.ones(6), [200]])
    c = base.c.copy()
    c[7:9] = c.max() * 50
    check(W.Network(60, 2900, base.reac_rxn, base.reac_sp, base.reac_coef, rxn, sp, d, c), W.poisson_x0(60, 30, 1),
          ctas_per_traj=ctas)


@pytest.mark.parametrize("m,ctas", [(1, 1), (33, 2), (1025, 1), (1025, 7), (5001, 152), (5001, 0)])
def test_one_channel_again_and_again(m, ctas):
    net = W.pure_birth(3.0) if m == 1 else W.random_mass_action(max(2, m // 8), m, 3 + m, 0.3)
    c = np.full(m, 1e-9)
    c[(2 * m) // 3] = 5.0
    check(net.with_rates(c), np.full(net.n_species, 400, np.int32), max_events=300, ctas_per_traj=ctas)


def test_overflow_is_not_fired():
    m = 300
    base = W.random_mass_action(40, m, 12, 0.5)
    c = np.full(m, 1e-12)
    k = int(base.stoi_rxn[base.stoi_delta > 0][0])
    s = int(base.stoi_sp[base.stoi_delta > 0][0])
    c[k] = 1.0
    x0 = np.full(40, 1000, np.int32)
    x0[s] = 2**31 - 5
    o = check(base.with_rates(c), x0, max_events=50, ctas_per_traj=2)
    assert (o["status"] == oracle.ST_OVERFLOW).any() or (o["n_events"] > 0).any()


@pytest.mark.parametrize("ctas", [2, 32, 33, 65, 152])
def test_every_lane_reads_the_partials_of_its_event(ctas):
    """One, several or no partial minima per lane, exchanged a few thousand times: a lane that read a partial
    of an earlier event would leave the oracle's path."""
    net = W.random_mass_action(600, 152 * 32, 77, 1.0)
    check(net, W.poisson_x0(600, 40, 5), n_traj=1 if ctas > 76 else 2, max_events=2000, ctas_per_traj=ctas)


def test_every_trajectory_stops_at_the_range_check():
    """One channel fires up to the last count that fits and is not fired past it, in every trajectory."""
    m = 300
    base = W.random_mass_action(40, m, 12, 0.5)
    c = np.full(m, 1e-12)
    k = int(base.stoi_rxn[base.stoi_delta > 0][0])
    s = int(base.stoi_sp[base.stoi_delta > 0][0])
    c[k] = 1.0
    x0 = np.full(40, 1000, np.int32)
    x0[s] = 2**31 - 5
    o = check(base.with_rates(c), x0, max_events=50, ctas_per_traj=2)
    assert (o["status"] == oracle.ST_OVERFLOW).all()
    assert (o["n_events"] > 0).all() and (o["n_events"] < 50).all()
