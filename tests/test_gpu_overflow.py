"""Layer buffers that run over while other streams keep the GPU busy: the warps of
a launch start at different times, some after the overflow is already noted."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import os, sys
sys.path.insert(0, '.')
import torch
from paper_2012_07620_gb300 import rerank
g = torch.Generator().manual_seed(2)
jobs = []
for k in range(24):
    n = 2500 + 40 * k
    x = (torch.randn(n // 12, 64, generator=g)[torch.randint(n // 12, (n,), generator=g)]
         + 0.9 * torch.randn(n, 64, generator=g)).cuda()
    jobs.append(dict(xq=x[:300].contiguous(), xg=x[300:].contiguous(), k1=26, k2=8, layers=3))
with rerank.Reranker(precision='bf16') as F:
    want = [F.run(j['xq'], j['xg'], 26, 8, 3) for j in jobs]
os.environ['RERANK_TEST_CAP_H'] = '90000'   # below every layer's need
with rerank.Reranker(precision='bf16') as R:
    got = R.run_batch(jobs)
    assert R.batch_status == [0] * len(jobs)
    torch.cuda.synchronize()
for (i, d), (wi, wd) in zip(got, want):
    assert torch.equal(i, wi) and torch.equal(d, wd)
print('ok')
"""


def test_overflow_under_other_streams():
    import __graft_entry__
    __graft_entry__.build()
    r = subprocess.run([sys.executable, "-c", CHILD], capture_output=True, text=True, timeout=600, cwd=ROOT)
    assert r.returncode == 0 and "ok" in r.stdout, (r.stdout[-2000:], r.stderr[-2000:])
