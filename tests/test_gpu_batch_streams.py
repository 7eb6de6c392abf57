"""The number of streams of a batch: what the library says it runs, one candidate
for counts that are the same, and a process with more hardware queues."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu


def _run(code, queues):
    env = {k: v for k, v in os.environ.items() if k != "CUDA_DEVICE_MAX_CONNECTIONS"}
    if queues:
        env["CUDA_DEVICE_MAX_CONNECTIONS"] = str(queues)
    r = subprocess.run([sys.executable, "-c", code], env=env, capture_output=True, text=True, timeout=300,
                       cwd=os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
    assert r.returncode == 0, r.stdout + r.stderr


@pytest.mark.parametrize("queues,most", [(None, 8), (20, 20), (32, 32), (33, 8)])
def test_streams_that_run(queues, most):
    _run(f"""
import os
import paper_1911_11906_gb300 as F
ctx = F.Context()
os.environ["CUDA_DEVICE_MAX_CONNECTIONS"] = "3"  # not what the device's queues were made with
for asked, count in ((0, 100), (4, 100), (16, 100), (32, 100), (64, 100), (64, 5), (1, 0)):
    want = max(1, min(asked or 16, count, 64, {most}))
    assert ctx.batched_workers(asked, count) == want, (asked, count)
""", queues)


def test_the_tuner_times_a_number_of_streams_once(tmp_path):
    _run(f"""
import json, torch
import paper_1911_11906_gb300 as F
from paper_1911_11906_gb300 import autotune as A
probs = [{{"A": torch.diag(torch.arange(1.0, 25.0 + i, dtype=torch.float64, device="cuda"))}} for i in range(40)]
path = {str(tmp_path / "tune.json")!r}
w = A.best_workers(probs, candidates=(4, 8, 16, 32), tuner=A.Autotuner(path))
(val,) = [v for k, v in json.load(open(path))["entries"].items() if k.startswith("batched_workers:")]
assert set(val["seconds"]) == {{"4", "8"}} and w in (4, 8)
""", None)


def test_fp64_panels_of_workers_with_few_sms():
    """20 streams or more leave a worker 8 SMs or fewer: FP64 panels of more than 256
    rows a CTA, in a batch after one whose workers had all 16 (tolerance 10 n eps)."""
    _run("""
import torch
import paper_1911_11906_gb300 as F
ctx = F.Context(wait_timeout_s=5.0)
g = torch.Generator(device="cuda").manual_seed(1)
def problem(n):
    A = torch.randn(n, n, dtype=torch.float64, device="cuda", generator=g)
    return {"A": A + A.t()}
def check(p, out):
    A, (lam, V, _) = p["A"], out
    n, eps = A.shape[0], torch.finfo(torch.float64).eps
    assert (V.t() @ V - torch.eye(n, dtype=torch.float64, device="cuda")).norm() <= 10 * n * eps
    assert (A @ V - V * lam).norm() <= 10 * n * eps * A.norm()
    assert ctx.batched_workers(32, 24) == 24
for count, n in ((1, 300), (24, 2800), (24, 4200)):
    probs = [problem(n)] + [problem(40 + i) for i in range(count - 1)]
    for p, o in zip(probs, F.solve_batched(probs, workers=32, ctx=ctx)):
        check(p, o)
""", 32)
