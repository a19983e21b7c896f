"""The clustered LM head, whose W loads multicast, is for programs on one GPU:
bench.py's replicas refuse every workload that could take it, and the library
chooses it only where the process sees a single GPU and W is that GPU's memory.
The latter on the CPU, with the three runtime queries that decide it replaced
by a small library loaded in front of the CUDA runtime."""
import os
import shutil
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
LIB = os.path.join(ROOT, "paper_2609_02897_gb300", "_lib", "libasd.so")


@pytest.mark.parametrize("argv", [["--config", "3"], ["--batch", "5"], ["--batch", "1"],
                                  ["--config", "2", "--batch", "64"], ["--config", "5", "--batch", "8"]])
def test_replicas_run_the_headline_workload_only(monkeypatch, argv):
    monkeypatch.syspath_prepend(ROOT)
    import bench
    for name in ("run_asd", "run_reference"):
        monkeypatch.setattr(bench, name, lambda args: pytest.fail("the workload was run"))
    monkeypatch.setattr(sys, "argv", ["bench.py", "--gpus", "2"] + argv)
    monkeypatch.setenv("WORLD_SIZE", "2")
    with pytest.raises(SystemExit, match="only the headline workload"):
        bench.main()


def test_replicas_of_the_headline_workload_run(monkeypatch):
    monkeypatch.syspath_prepend(ROOT)
    import bench
    ran = []
    monkeypatch.setattr(bench, "run_asd", ran.append)
    monkeypatch.setattr(sys, "argv", ["bench.py", "--gpus", "2"])
    monkeypatch.setenv("WORLD_SIZE", "2")
    bench.main()
    assert len(ran) == 1


QUERIES = r"""
#include <string.h>
int gpus;              /* visible GPUs */
int owner;             /* the GPU that W belongs to */
int cudaGetDeviceCount(int* n) { *n = gpus; return 0; }
int cudaGetDevice(int* d) { *d = 0; return 0; }
int cudaDeviceGetAttribute(int* v, int attr, int dev) { (void)attr; (void)dev; *v = 152; return 0; }
/* cudaPointerAttributes: type (2: device memory), device, two pointers */
int cudaPointerGetAttributes(int* a, const void* p) {
  (void)p; memset(a, 0, 8); a[0] = 2; a[1] = owner; return 0;
}
"""

ASK = r"""
import ctypes, sys
q = ctypes.CDLL(sys.argv[1], mode=ctypes.RTLD_GLOBAL)
lib = ctypes.CDLL(sys.argv[2])
ctypes.c_int.in_dll(q, "gpus").value = int(sys.argv[3])
ctypes.c_int.in_dll(q, "owner").value = int(sys.argv[4])
lib.asd_lm_head_variant.argtypes = [ctypes.c_void_p, ctypes.c_int32, ctypes.c_void_p]
# batch, heads, KV heads, D, hidden, vocab, bf16, page, cache, pages, nodes, path, layout, rule, schedule
dims = (ctypes.c_int32 * 15)(8, 32, 8, 128, 4096, 128256, 1, 0, 64, 0, 128, 8, 0, 0, 0)
print([lib.asd_lm_head_variant(dims, t, 4096) for t in (60, 256, 384, 512, 640, 896, 1024)])
"""


@pytest.mark.skipif(shutil.which("gcc") is None, reason="needs a C compiler")
@pytest.mark.parametrize("gpus,owner,want", [(1, 0, [1, 2, 3, 3, 2, 3, 3]), (2, 0, [1, 2, 2, 2, 2, 2, 2]),
                                             (8, 0, [1, 2, 2, 2, 2, 2, 2]), (1, 1, [1, 2, 2, 2, 2, 2, 2])])
def test_the_library_multicasts_on_a_single_gpu_only(tmp_path, gpus, owner, want):
    src, so = tmp_path / "queries.c", tmp_path / "libqueries.so"
    src.write_text(QUERIES)
    subprocess.run(["gcc", "-shared", "-fPIC", "-o", str(so), str(src)], check=True)
    # where the loader finds the CUDA runtime: next to the one that torch loads
    import torch  # noqa: F401
    with open("/proc/self/maps") as f:
        dirs = {os.path.dirname(line.split()[-1]) for line in f if "libcudart" in line}
    env = dict(os.environ, LD_LIBRARY_PATH=":".join(sorted(dirs) + [os.environ.get("LD_LIBRARY_PATH", "")]))
    out = subprocess.run([sys.executable, "-c", ASK, str(so), LIB, str(gpus), str(owner)], env=env,
                         capture_output=True, text=True, check=True).stdout
    assert out.strip() == str(want)
