"""nr_render_static allocates nothing: neither device nor pinned host memory, in a subject's first
call as in any later one.  The runtime's allocation calls are counted by a small library loaded
ahead of it, in a process of its own."""
import os
import shutil
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

COUNTER = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stddef.h>
static int calls;
int allocation_calls(void) { return calls; }
static void *real(const char *name) {
  void *rt = dlopen("libcudart.so.13", RTLD_LAZY | RTLD_NOLOAD);
  return rt ? dlsym(rt, name) : NULL;
}
#define COUNTED(name, params, args)                                       \
  int name params {                                                       \
    int (*fn) params = (int (*) params)real(#name);                       \
    __atomic_add_fetch(&calls, 1, __ATOMIC_SEQ_CST);                      \
    return fn ? fn args : 3;                                              \
  }
COUNTED(cudaMalloc, (void **p, size_t n), (p, n))
COUNTED(cudaMallocHost, (void **p, size_t n), (p, n))
COUNTED(cudaHostAlloc, (void **p, size_t n, unsigned f), (p, n, f))
COUNTED(cudaMallocManaged, (void **p, size_t n, unsigned f), (p, n, f))
COUNTED(cudaMallocAsync, (void **p, size_t n, void *s), (p, n, s))
COUNTED(cudaHostRegister, (void *p, size_t n, unsigned f), (p, n, f))
"""

SCRIPT = r"""
import ctypes, sys
sys.path.insert(0, sys.argv[2])
import numpy as np, torch
from paper_2306_16541_gb300 import nr, synth
count = ctypes.CDLL(sys.argv[1]).allocation_calls
s = synth.subject(421, hash_scale=0.5, res_last_std=0.02, with_ellipsoids=True)
pose = synth.random_pose(np.random.default_rng(422))
cam = nr.make_camera(synth.camera(32, 32, 40.0, (0.0, 0.0, 2.5), 32, 1.5, 3.5))
out = torch.empty(32, 32, 4, device="cuda")
for mlp, kw in (("bf16", {}), ("f16", {}), ("bf16", dict(tcgen05=True)), ("bf16", dict(mma2=True)), ("f32", {})):
    for t_min in (0.0, 1e-4):
        o = nr.make_opts(mlp, "f32" if mlp == "f32" else "f16", t_min == 0.0, t_min, **kw)
        n0 = count()
        S = nr.Subject(s)
        S.set_pose(*pose)
        torch.cuda.synchronize()
        n1 = count()
        assert n1 > n0, "the counter does not see the library's calls"
        for _ in range(2):
            nr.nr_render_static(S.h, cam, o, out)
        torch.cuda.synchronize()
        n2 = count()
        S.close()
        print(mlp, kw, t_min, n2 - n1)
        assert n2 == n1, (mlp, kw, t_min, n2 - n1)
print("allocation-free")
"""


def test_the_first_static_render_of_a_subject_allocates_nothing(tmp_path):
    cc = shutil.which("gcc") or shutil.which("cc")
    if not cc:
        pytest.skip("no C compiler")
    from paper_2306_16541_gb300 import build
    build.build()
    src, lib = tmp_path / "count.c", tmp_path / "count.so"
    src.write_text(COUNTER)
    subprocess.run([cc, "-shared", "-fPIC", "-O1", "-o", str(lib), str(src), "-ldl"], check=True)
    p = subprocess.run([sys.executable, "-c", SCRIPT, str(lib), ROOT], cwd=ROOT, capture_output=True, text=True,
                       timeout=300, env=dict(os.environ, LD_PRELOAD=str(lib)))
    assert p.returncode == 0 and "allocation-free" in p.stdout, p.stdout + p.stderr
