"""The weight-gradient kernel where no tensor map can be made.

The driver's encode function is found at run time.  Where it is not, the calls
that need the kernel report RC_ECUDA, the timed step among them (its phases would
leave the weight gradients out), and the mma.sync engine, which needs no tensor
map, still runs.  The entry-point query is faked in a child process.
"""
import os
import shutil
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

FAKE = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
#include <string.h>
typedef int (*query)(const char *, void **, unsigned, unsigned long long, int *);
int cudaGetDriverEntryPointByVersion(const char *name, void **fn, unsigned version, unsigned long long flags, int *q) {
    if (!strcmp(name, "cuTensorMapEncodeTiled")) return 500; /* not found */
    void *rt = dlopen("libcudart.so.13", RTLD_LAZY);
    return ((query)dlsym(rt, "cudaGetDriverEntryPointByVersion"))(name, fn, version, flags, q);
}
"""

CHILD = """
import numpy as np, torch
from paper_1902_09171_gb300 import rcell, surrogate as S
torch.cuda.set_device(0)
rcell.load()
s = S.sur_create(2, 64, 4, 0)
U, Y = torch.zeros(20, 3, 15, device="cuda"), torch.ones(20, 3, 6, device="cuda")
for backend in (2, 1, 0):
    S.sur_set_backend(s, backend)
    for call in (lambda: S.sur_loss_grad(s, 0, U, Y), lambda: S.sur_train_step(s, U, Y, 1e-3, n_members=2),
                 lambda: S.sur_profile_step(s, U, Y)):
        try:
            call()
            print("ok", end=" ")
        except rcell.RCellError as e:
            print(e.name, end=" ")
assert S.sur_sync(s) == 0
S.sur_destroy(s)
"""


def test_calls_without_tensor_maps_say_so(tmp_path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    cc = shutil.which("gcc") or shutil.which("cc")
    if not cc:
        pytest.skip("no C compiler")
    from paper_1902_09171_gb300 import build
    build.build()
    src, lib = tmp_path / "fake.c", tmp_path / "libfake.so"
    src.write_text(FAKE)
    subprocess.run([cc, "-shared", "-fPIC", "-o", str(lib), str(src), "-ldl"], check=True)
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, capture_output=True, text=True, timeout=300,
                       env=dict(os.environ, LD_PRELOAD=str(lib)))
    assert r.returncode == 0, r.stderr
    assert r.stdout.split() == ["RC_ECUDA"] * 6 + ["ok"] * 3
