"""A solver whose guided rounds' mirror finds no memory: cudaMallocAsync is
replaced, for allocations of the mirror's size, by one that refuses."""
import json
import os
import subprocess
import sys

import numpy as np
import pytest

import lbdd_inputs as L
import oracle

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SHIM = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stdio.h>
#include <stdlib.h>
int cudaMallocAsync(void** p, size_t n, void* stream) {
  static int (*real)(void**, size_t, void*);
  const size_t lo = strtoull(getenv("REFUSE_LO"), 0, 10), hi = strtoull(getenv("REFUSE_HI"), 0, 10);
  if (!real) {
    void* rt = dlopen("libcudart.so.13", RTLD_LAZY | RTLD_NOLOAD);
    real = (int (*)(void**, size_t, void*))dlsym(rt, "cudaMallocAsync");
  }
  if (n >= lo && n < hi) { fprintf(stderr, "refused %zu\n", n); return 2; }
  return real(p, n, stream);
}
"""

CHILD = """
import json, sys
import numpy as np
import lbdd_inputs as L
import paper_2304_06543_gb300 as lb
lib = lb.load()
inst = L.random_small(9500, n=300, k=400, cm_max=50, cap_frac=0.5, pen=(5, 60))
with lb.Solver(inst.cm.astype(np.int16), inst.cap, inst.pen) as s:
    s.solve()
    print(json.dumps({"objective": s.objective, "guided": s.guided_rounds, "assign": s.assignment().tolist(),
                      "error": lib.lbdd_last_cuda_error().decode()}))
"""


def test_mirror_without_memory(gpu_lib, tmp_path):
    k = 400
    src, so = tmp_path / "refuse.c", tmp_path / "refuse.so"
    src.write_text(SHIM)
    subprocess.run(["gcc", "-shared", "-fPIC", "-o", str(so), str(src), "-ldl"], check=True)
    # the mirror: k rows of k to k + 8 int16 costs; no other array has that size
    env = dict(os.environ, LD_PRELOAD=str(so), REFUSE_LO=str(2 * k * k),
               REFUSE_HI=str(2 * k * (k + 8) + 1), PYTHONPATH=ROOT)
    out = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, env=env, capture_output=True,
                         text=True, timeout=300)
    assert out.returncode == 0, out.stderr
    assert out.stderr.count("refused") == 1, out.stderr
    got = json.loads(out.stdout.strip().splitlines()[-1])
    inst = L.random_small(9500, n=300, k=k, cm_max=50, cap_frac=0.5, pen=(5, 60))
    ref = oracle.asral(inst.cm, inst.cap, inst.pen)
    assert ref.stats["moves"] > 0
    assert got["objective"] == ref.delta and np.array_equal(got["assign"], ref.assign)
    assert got["error"] == "no error" and got["guided"] == 0
