"""A CUDA call that fails inside a step is reported: the maximum of the current histogram
(pauli_norm = 1) starts with a memset, whose error a step that ignored it would hide while its Pauli
test ran against a stale or zero maximum.  The failure is an error code from a preloaded stand-in for
cudaMemsetAsync, in a process of its own; nothing invalid reaches the device."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SHIM = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stddef.h>
int shim_fail = 0, shim_calls = 0;
int cudaMemsetAsync(void *p, int v, size_t n, void *s)
{
    static int (*real)(void *, int, size_t, void *);
    if (shim_fail) { ++shim_calls; return 1; }
    if (!real) {
        void *h = dlopen("libcudart.so.13", RTLD_LAZY | RTLD_NOLOAD);
        real = (int (*)(void *, int, size_t, void *))(h ? dlsym(h, "cudaMemsetAsync") : NULL);
    }
    return real ? real(p, v, n, s) : 999;
}
"""

CHILD = r"""
import ctypes, sys
sys.path.insert(0, sys.argv[2])
import torch
from paper_2404_19602_gb300 import pgc, workloads as W
sim = pgc.Simulation(W.scaled(W.DET_FP64_1E4, N=1000, pauli_norm=1, precision=sys.argv[3]), max_outputs=4)
sim.set_pipeline(sys.argv[4] == "1")
sim.step(2)
torch.cuda.synchronize()
shim = ctypes.CDLL(sys.argv[1])
ctypes.c_int.in_dll(shim, "shim_fail").value = 1
try:
    sim.step(1)
    print("returned", ctypes.c_int.in_dll(shim, "shim_calls").value)
except pgc.PgcError as e:
    print("raised", ctypes.c_int.in_dll(shim, "shim_calls").value)
ctypes.c_int.in_dll(shim, "shim_fail").value = 0
"""


@pytest.mark.parametrize("precision,pipeline", [("fp32", "0"), ("fp64", "1")])
def test_failed_memset_of_the_maximum_is_reported(tmp_path, precision, pipeline):
    from paper_2404_19602_gb300 import build

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    src, lib = str(tmp_path / "shim.c"), str(tmp_path / "shim.so")
    open(src, "w").write(SHIM)
    subprocess.run(["gcc", "-shared", "-fPIC", "-O1", "-o", lib, src, "-ldl"], check=True)
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", CHILD, lib, root, precision, pipeline], capture_output=True, text=True,
                       timeout=240, env=dict(os.environ, LD_PRELOAD=lib))
    assert r.returncode == 0, r.stderr[-2000:]
    assert r.stdout.split() == ["raised", "1"], r.stdout
