"""First launches of the prologue's kernels in a process.

A kernel's dynamic shared memory beyond the 48 KB default needs an opt-in per kernel, and the default covers the kernel's
static part too.  The sizes here lie just below 48 KB of dynamic memory, each the first call of its kernel in a fresh process,
where no wider call before it has raised the limit."""
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

# input type, rows, channels, group size, dynamic positions: ring of whole rows (static, dynamic beyond the one-launch
# kernel's 10 MB), then the one-launch dynamic kernel at 767 rows per CTA
CASES = [("float32", 400, 1520, 16, False), ("float16", 300, 5920, 16, False), ("bfloat16", 300, 5952, 16, False), ("int8", 300, 9280, 16, False),
         ("float32", 2000, 1344, 16, True), ("float16", 4000, 1344, 16, True), ("bfloat16", 6200, 1152, 16, True), ("int8", 1600, 6656, 32, True),
         ("float32", 6130, 64, 64, True), ("float16", 6129, 64, 64, True), ("bfloat16", 6136, 64, 64, True), ("int8", 6133, 64, 64, True)]

CHILD = """
import torch
from paper_2510_02822_b200 import binding as fx
for kind, M, K, G, dynamic in {cases!r}:
    q = (torch.arange(M * K, device="cuda") * 7919 % 251 - 125).to(torch.int8).view(M, K)
    X = q if kind == "int8" else q.to(getattr(torch, kind)) * 0.25
    L = fx.Layer(torch.ones((K, 16), dtype=torch.int8, device="cuda"), torch.ones(16, device="cuda"), None, range(K // G), None, G)
    x4, _, _ = L.quantize_lower(X, 0.25, dynamic=dynamic)
    assert torch.equal(x4[:M * K].view(torch.int8).view(M, K), q), (kind, M, K, G, dynamic)
    fx.flexiq_check_status()
    L.close()
print("all first launches ok")
"""


def test_first_launches_of_a_process():
    r = subprocess.run([sys.executable, "-c", CHILD.format(cases=CASES)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "all first launches ok" in r.stdout, r.stderr[-2000:]
