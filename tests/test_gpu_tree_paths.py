"""The tree kernel's variants: every cluster size, networks whose net changes do not fit the packed
dependency records (more than four species, large changes), event lists that do not fit packed (each channel
once per reader list) beside those that do, one channel firing again and again, and groups at the end of a
slice.  All comparisons are exact."""
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

KEYS = ("x_final", "n_events", "status", "counts", "t_last", "t_internal", "loglik", "trace_mu", "trace_t")


def check(net, x0, n_traj=3, max_events=250, grad=True, **kw):
    g = api.simulate(api.Network(net), x0, 1e6, n_traj, seed=5, max_events=max_events, grad=grad, trace_len=max_events,
                     form=L.RT_FORM_ABSOLUTE, **kw)
    o = oracle.run(net, x0, 1e6, n_traj, seed=5, max_events=max_events, want_grad=grad, trace_len=max_events, mode=1,
                   n_threads=4)
    for k in KEYS:
        if k in g and k in o:
            a = g[k].cpu().numpy()
            b = o[k].astype(a.dtype)
            a, b = (a.view(np.int64), b.view(np.int64)) if a.dtype == np.float64 else (a, b)
            assert np.array_equal(a, b), k


@pytest.mark.parametrize("ctas", [1, 2, 4, 8, 16])
@pytest.mark.parametrize("m,n", [(700, 50), (4100, 90)])
def test_cluster_sizes(m, n, ctas):
    check(W.random_mass_action(n, m, 20 + m, 0.8), W.poisson_x0(n, 30, m), ctas_per_traj=ctas, grad=ctas != 2)


@pytest.mark.parametrize("ctas", [1, 4])
def test_records_that_do_not_pack(ctas):
    base = W.random_mass_action(60, 900, 4, 0.8)
    # reaction 7 also makes six other species, reaction 8 two hundred molecules of one
    rxn = np.concatenate([base.stoi_rxn, np.full(6, 7), [8]])
    sp = np.concatenate([base.stoi_sp, np.arange(40, 46), [50]])
    d = np.concatenate([base.stoi_delta, np.ones(6), [200]])
    c = base.c.copy()
    c[7:9] = c.max() * 20
    net = W.Network(60, 900, base.reac_rxn, base.reac_sp, base.reac_coef, rxn, sp, d, c)
    check(net, W.poisson_x0(60, 30, 1), ctas_per_traj=ctas)


@pytest.mark.parametrize("m,n", [(4000, 2), (2500, 3), (1200, 1)])
def test_dense_dependencies(m, n):
    """Every event touches most channels: the packed list does not fit for the largest of these."""
    check(W.random_mass_action(n, m, 6, 0.5), W.poisson_x0(n, 40, 3), n_traj=2, max_events=60, ctas_per_traj=1)


def test_one_channel_again_and_again():
    net = W.random_mass_action(20, 300, 3, 0.3)
    c = np.full(300, 1e-9)
    c[137] = 5.0
    check(net.with_rates(c), np.full(20, 500, np.int32), max_events=400)
    check(W.pure_birth(3.0), np.zeros(1, np.int32), max_events=300)


def _list_bytes(net, ctas):
    """Shared memory of a slice with the event's list of touched channels once per channel and once per reader
    list, from the sizes the kernel's plan is made of (16 bytes a group, 40 an entry, X)."""
    readers = np.bincount([s for _, s in set(zip(net.reac_rxn.tolist(), net.reac_sp.tolist()))],
                          minlength=net.n_species)
    change = {}
    for r, s, d in zip(net.stoi_rxn.tolist(), net.stoi_sp.tolist(), net.stoi_delta.tolist()):
        change[r, s] = change.get((r, s), 0) + d
    dep = np.zeros(net.n_reactions, np.int64)
    for (r, s), d in change.items():
        if d:
            dep[r] += readers[s]
    chunk = (-(-net.n_reactions // ctas) + 31) // 32 * 32
    most = int(dep.max())
    assert api.Network(net).info()["max_dependents"] == most
    return [chunk // 32 * 16 + cap * 40 + net.n_species * 4 for cap in (min(chunk, most + 1), min(2 * chunk, most) + 1)]


@pytest.mark.parametrize("m,n,ctas", [(4400, 2, 1), (4900, 3, 1), (9000, 2, 2)])
def test_list_that_fits_once_per_channel_only(m, n, ctas):
    """Networks so dense that an event's list has no room for a channel found in two reader lists: each channel is
    updated where it is found and takes its entry there."""
    net = W.random_mass_action(n, m, 6, 0.5)
    once, twice = _list_bytes(net, ctas)
    assert once <= 200 * 1024 < twice
    check(net, W.poisson_x0(n, 40, 3), n_traj=2, max_events=80, ctas_per_traj=ctas, grad=ctas == 1)
