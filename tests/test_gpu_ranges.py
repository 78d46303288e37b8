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
