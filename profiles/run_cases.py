"""Runs cases of perf/cases.py once each, for a profiler: python profiles/run_cases.py CASE...  (from the repository's root)

A name may be followed by ":lse": the row log-sum-exp first, then kvm_score with it, whose column pass carries no similarities.
"""
import os
import sys

import torch

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import paper_2407_08454_b200 as kvm  # noqa: E402
from perf import cases  # noqa: E402

by_name = {c["name"]: c for c in cases.listed()}
for arg in sys.argv[1:]:
    name, _, form = arg.partition(":")
    st = cases.prepare(by_name[name], 1)
    if form == "lse":
        Q, K, ws = st["Q"], st["K"], st["comp"].ws
        lse, scores = (torch.empty(t.shape[:3], dtype=torch.float32, device="cuda") for t in (Q, K))
        kvm.kvm_row_lse(st["p"], Q, K, lse, ws)
        kvm.kvm_score(st["p"], Q, K, lse, scores, ws)
    else:
        cases.run(st)
    torch.cuda.synchronize()
    del st
