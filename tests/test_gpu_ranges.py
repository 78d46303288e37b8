"""Edges of the integer arithmetic on the simulation path, against the oracle bit for bit: the
table-driven logarithm at the edges of its buckets and around the values where it hands over to the
series, and whole trajectories whose rates leave the range of the float estimates and of the integer
division and product (which then use the FP64 pipe).  Equality is exact: both sides define the same bits.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_2103_00405_gb300 import workloads as W

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - CPU-only hosts skip the GPU suite
    pytest.skip("CUDA not available", allow_module_level=True)

from paper_2103_00405_gb300 import api  # noqa: E402


def test_log_at_the_bucket_edges():
    k = np.arange(64, 129)[:, None] / 128.0
    near = (k * (1 + np.arange(-6, 7)[None] * 2.0**-53)).ravel()
    half = np.sqrt(0.5) * (1 + np.arange(-40, 41) * 2.0**-53)
    fine = 1 - np.arange(1, 70) / 4096.0
    base = np.concatenate([near, half, fine, fine * (1 - 2.0**-50), 1 - 2.0**-np.arange(1, 53)])
    x = np.concatenate([np.ldexp(base, e) for e in (-1022, -53, -1, 0, 1, 2, 3, 40, 1000)])
    y = api.log_eval(torch.from_numpy(x).cuda()).cpu().numpy()
    lib = oracle.load()
    ref = np.array([lib.oracle_rt_log(float(v)) for v in x])
    assert np.array_equal(y.view(np.int64), ref.view(np.int64))


def test_draws_equal_the_oracle_over_many_indices():
    n = 150000
    idx = np.arange(n, dtype=np.uint64)
    u, e = api.draw_exp1(12345, np.full(n, 3, np.uint64), np.full(n, 7, np.uint32), idx)
    lib = oracle.load()
    ref = np.array([lib.oracle_exp1(12345, 3, 7, int(i), 0) for i in range(n)])
    assert np.array_equal(e.cpu().numpy().view(np.int64), ref.view(np.int64))


@pytest.mark.parametrize("scale", [1e-310, 1e-200, 1e-37, 1e37, 1e200])
@pytest.mark.parametrize("m,n", [(1, 1), (3, 2), (4, 4), (7, 6), (14, 7), (40, 10), (600, 60)])
def test_rates_outside_the_float_range(m, n, scale):
    """Every second rate scaled far out: estimates, products and quotients at and beyond their ranges."""
    net = W.pure_birth() if m == 1 else W.random_mass_action(n, m, 900 + m, 0.5)
    c = net.c.copy()
    c[::2] *= scale
    net = net.with_rates(c)
    x0 = np.full(net.n_species, 40, np.int32)
    g = api.simulate(api.Network(net), x0, 1e300, 5, seed=3, max_events=150, grad=True)
    o = oracle.run(net, x0, 1e300, 5, seed=3, max_events=150, want_grad=True, n_threads=4)
    for key in ("x_final", "n_events", "status", "counts"):
        assert np.array_equal(g[key].cpu().numpy(), o[key]), key
    for key in ("t_last", "t_internal", "loglik"):
        a, b = g[key].cpu().numpy(), o[key]
        assert ((a.view(np.int64) == b.view(np.int64)) | (np.isnan(a) & np.isnan(b))).all(), key
