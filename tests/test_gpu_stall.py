"""Waits that run out in every epilogue of the tensor-core kernels (sampling,
append, lists on pairs, lists on single CTAs): ETIMEOUT, and the context goes on.
Sizes are past 1,024 rows, where the sampling pass runs."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import os, sys
sys.path.insert(0, '.'); sys.path.insert(0, 'tests')
import torch
import parity
from oracle import rerank_oracle as o
from paper_2012_07620_gb300 import rerank, synthetic
w = synthetic.make_workload(synthetic.WorkloadSpec('stall', 60, 1440, 128, 80, 0.35, 0, None, seed=3))
xq, xg = torch.from_numpy(w.xq).cuda(), torch.from_numpy(w.xg).cuda()
precision, lists = sys.argv[1], sys.argv[2] == 'lists'
budget = 0
if lists:  # a budget below the append plan
    del os.environ['RERANK_TEST_TC_STALL']
    with rerank.Reranker(precision=precision) as F:
        F.run(xq, xg, 26, 7, 2)
        budget = F.last_info()['workspace_bytes'] * 8 // 9 - (1 << 20)
    os.environ['RERANK_TEST_TC_STALL'] = '1'
with rerank.Reranker(precision=precision, hbm_budget=budget) as R:
    try:
        R.run(xq, xg, 26, 7, 2)
        sys.exit('returned without error')
    except rerank.RerankError as e:
        assert e.status == 5, e.status
    del os.environ['RERANK_TEST_TC_STALL']
    i, d = R.run(xq, xg, 26, 7, 2)
    torch.cuda.synchronize()
    if lists:
        assert R.last_info()['candidates_per_row'] == 42
ref = o.rerank(w.xq, w.xg, 26, 7, 2, mode='sparse')
parity.assert_ranked_equal(i.cpu().numpy(), d.cpu().numpy(), ref.s, ref.idx)
print('ok')
"""


@pytest.mark.parametrize("precision,plan,pairs", [("bf16", "append", "1"), ("fp8", "append", "1"),
                                                  ("bf16", "lists", "1"), ("bf16", "append", "0")])
def test_waits_of_every_epilogue_run_out(precision, plan, pairs):
    import __graft_entry__
    __graft_entry__.build()
    env = dict(os.environ, RERANK_TEST_TC_STALL="1", RERANK_TC_PAIRS=pairs)
    r = subprocess.run([sys.executable, "-c", CHILD, precision, plan], env=env, capture_output=True, text=True,
                       timeout=600, cwd=ROOT)
    assert r.returncode == 0 and "ok" in r.stdout, (r.stdout[-2000:], r.stderr[-2000:])
