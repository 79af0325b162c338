"""Contexts are independent: host threads, each with a context of its own, whose calls need
different amounts of the same kernels' shared memory."""
import os
import subprocess
import sys
import threading

import numpy as np
import pytest

from paper_2609_02109_gb300 import workload as W

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def mf():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2609_02109_gb300 import mf as m
    return m


def _same(a, b):
    return all(np.array_equal(a[f], b[f]) for f in ("topk_idx", "topk_score", "count"))


@pytest.mark.parametrize("call", ["search_fp32", "search_bf16", "fc_search", "fc_ga"])
def test_threads_with_lists_of_their_own_size(mf, call):
    import torch
    prob = W.make_problem([9, 8, 7], 8, 32, 0, 3, 40.0, precision="bf16" if call == "search_bf16" else "fp32")
    fc = W.fc_scenario(prob, 3)

    def run(ctx, k):
        if call == "fc_search":
            return ctx.fc_search(k)
        if call == "fc_ga":
            fit, genome = ctx.fc_ga_run(dict(W.PAPER_GA_PARAMS, pop=k, gens=2), 5)
            return dict(topk_idx=genome, topk_score=fit, count=0)
        return ctx.search(k)

    failed = []

    def worker(k):
        try:
            with torch.cuda.stream(torch.cuda.Stream()), mf.Context(prob) as ctx:
                ctx.fc_set(fc)
                want = run(ctx, k)
                gate.wait()
                for _ in range(300):
                    assert _same(run(ctx, k), want)
        except BaseException as e:  # noqa: BLE001  (reported below)
            gate.abort()
            failed.append((k, repr(e)))

    ks = [8] * 5 + [128 if call == "search_bf16" else 1000]
    gate = threading.Barrier(len(ks))
    threads = [threading.Thread(target=worker, args=(k,)) for k in ks]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed


# Stands before the runtime's own function and notes each value that a kernel's limit of
# dynamic shared memory (attribute 8) is set to; at exit, the kernels with more than one.
SHIM = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stdio.h>
static const void* func[256];
static int value[256], n, changed;
int cudaFuncSetAttribute(const void* f, int attr, int v) {
  int (*real)(const void*, int, int) = (int (*)(const void*, int, int))dlsym(RTLD_NEXT, "cudaFuncSetAttribute");
  int i = 0;
  while (attr == 8 && i < n && func[i] != f) ++i;
  if (attr == 8 && i == n && n < 256) { func[n] = f; value[n++] = v; }
  else if (attr == 8 && i < n && value[i] != v) ++changed;
  return real(f, attr, v);
}
__attribute__((destructor)) static void report(void) { fprintf(stderr, "limits set %d, changed %d\n", n, changed); }
"""

CALLS = """
from paper_2609_02109_gb300 import mf, workload as W
prob = W.make_problem([9, 8, 7], 8, 32, 0, 3, 40.0)
with mf.Context(prob) as ctx, mf.Context(prob, precision="bf16") as half:
    ctx.fc_set(W.fc_scenario(prob, 3))
    for k in (1000, 65, 8):
        ctx.search(k)
        ctx.fc_search(k)
        half.search(min(k, 128))
        ctx.fc_ga_run(dict(W.PAPER_GA_PARAMS, pop=k, gens=2), 5)
"""


def test_limits_do_not_depend_on_the_call(mf, tmp_path):
    """A kernel's limit of dynamic shared memory belongs to the process: a call that set it to
    its own need could fail another thread's launch that needs more."""
    (tmp_path / "shim.c").write_text(SHIM)
    shim = str(tmp_path / "shim.so")
    subprocess.run(["gcc", "-shared", "-fPIC", "-O1", "-o", shim, str(tmp_path / "shim.c"), "-ldl"], check=True)
    r = subprocess.run([sys.executable, "-c", CALLS], cwd=ROOT, env=dict(os.environ, LD_PRELOAD=shim),
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    said = [line for line in r.stderr.splitlines() if line.startswith("limits set ")]
    n, changed = (int(w) for w in said[-1].replace(",", "").split()[2::2])
    assert n >= 4 and changed == 0
