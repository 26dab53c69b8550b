"""Explicit inverses of the coarsest pixel levels where their memory cannot be
had: the allocation is refused on the host (a cudaMalloc preloaded before the
runtime's returns cudaErrorMemoryAllocation for one size), and the precompute
and a load go on with the sweeps."""
import os
import shutil
import subprocess
import sys

import pytest

from gpu_util import cuda_device

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

FAKE = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stdio.h>
#include <stdlib.h>
int cudaMalloc(void** p, size_t n) {
  static int (*next)(void**, size_t);
  const char* size = getenv("REFUSE_BYTES");
  if (size && n == strtoull(size, 0, 10)) {
    fprintf(stderr, "refused\n");
    return 2;
  }
  if (!next) next = (int (*)(void**, size_t))dlsym(RTLD_NEXT, "cudaMalloc");
  return next(p, n);
}
"""

RUN = r"""
import sys
import numpy as np
import torch
from paper_1308_5299_gb300 import binding, synthetic
cfg, cl, bl, ninv = synthetic.problem_inputs("nside32_lmax95")
kw = dict(nside=cfg["nside"], cl=cl, bl=bl, ninv=torch.from_numpy(ninv).cuda(), levels="default")
sweeps = binding.Plan(cfg["lmax"], smoother_sweep="cooperative", **kw)
ridges = [sweeps.level(h)["ridge"] for h in range(1, sweeps.nlevels() + 1)]
auto = binding.Plan(cfg["lmax"], ridge_alpha=ridges, **kw)
auto.save(sys.argv[1])
loaded = binding.Plan(cfg["lmax"], defer_precompute=True, ridge_alpha=ridges, **kw)
loaded.load(sys.argv[1])
for plan in (auto, loaded):
    for h in range(1, plan.nlevels() + 1):
        m = torch.from_numpy(synthetic.random_map(12 * plan.level(h)["nside_h"] ** 2, seed=h)).float().cuda()
        a, b = torch.empty_like(m), torch.empty_like(m)
        plan.pixel_smoother(h, m, a)
        sweeps.pixel_smoother(h, m, b)
        same = torch.equal(a, b)
        print(plan.level(h)["nside_h"], int(same), float((a - b).norm() / b.norm()))
"""


# (the panel of 12 tiles has the size of other buffers of the plan)
@pytest.mark.parametrize("what,tiles", [("inverse", 48), ("inverse", 12), ("panel", 48)])
def test_refused_inverse_leaves_the_sweeps(tmp_path, what, tiles):
    cuda_device()
    n = 64 * tiles
    size = 4 * n * n if what == "inverse" else 4 * 2 * 16 * n
    (tmp_path / "f.c").write_text(FAKE)
    cc = shutil.which("gcc") or "cc"
    subprocess.run([cc, "-shared", "-fPIC", "-o", str(tmp_path / "f.so"), str(tmp_path / "f.c"), "-ldl"], check=True)
    env = dict(os.environ, LD_PRELOAD=str(tmp_path / "f.so"), REFUSE_BYTES=str(size), PYTHONPATH=ROOT)
    r = subprocess.run([sys.executable, "-c", RUN, str(tmp_path / "c.bin")], cwd=ROOT, env=env, capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    assert "refused" in r.stderr
    rows = [x.split() for x in r.stdout.splitlines()]
    assert [int(x[0]) for x in rows] == [32, 16, 8] * 2
    for nside_h, same, err in rows:
        # the level whose memory was refused runs the very sweeps (as levels of more than 48 tiles do), the other
        # its inverse
        npix = 12 * int(nside_h) ** 2
        assert (same == "1") == (npix == n or npix > 48 * 64), rows
        assert float(err) < 2e-4
