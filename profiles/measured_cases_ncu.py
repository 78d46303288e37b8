"""Runs each case of perf/cases.py once at a size small enough for a capture with several passes (a few GB on the
device, launches of some ten milliseconds), from the repository's root:

    python profiles/measured_cases_ncu.py && ncu --metrics <a few> --clock-control none \
        -k 'regex:k_(ens|batch|bundle|lazy)' --csv --log-file launches.csv python profiles/measured_cases_ncu.py

Each line printed goes with one captured launch, in order (the initialisation kernels of the two large cases are
captured as well, k_bundle_init and k_lazy_init)."""
import os
import sys

sys.path.insert(0, os.getcwd())

import torch

import perf.cases as C
from paper_2103_00405_gb300 import api

REDUCED = {
    "bd_small_grid": {},
    "lv_64_paths": dict(t_end=0.5),
    "lv_ensemble": dict(n_traj=155648, t_end=0.1),
    "dimer_ensemble": dict(n_traj=311296),
    "small_model_m12": dict(n_traj=50000),
    "grad_m64": dict(n_traj=16384, max_events=1000),
    "pathway_m200": dict(max_events=1000),
    "network_m2000": dict(n_traj=304, max_events=1000),
    "batch_512": dict(max_events=2000),
    "large_internal": dict(max_events=60),
    "large_absolute": dict(max_events=1500),
    "ramped_m48": dict(max_events=300),
}

for case in C.listed():
    case = dict(case, **REDUCED[case["name"]])
    st = C.prepare(case, 5)
    if case["family"] == "grad":  # the forward launch alone
        net = api.Network(st["spec"])
        out = api.simulate(net, st["x0"], case["t_end"], case["n_traj"], seed=st["seed"],
                           max_events=case["max_events"], grad=True)
    else:
        out = C.run(st)
    torch.cuda.synchronize()
    print(case["name"], "events", int(out["n_events"].sum()), flush=True)
    del st, out
