"""Device memory that runs out while a schedule is prepared, or moved from the wavefronts to the class-major
arrays: no state is lost and nothing of the failed preparation is left behind.

The allocations are made to fail on the host, one after the other: the units that prepare schedules are
compiled a second time with their pool allocations going through a counter, and a child process runs on
that library.
"""
import concurrent.futures as cf
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
UNITS = ["sweep", "systolic", "stars", "stream"]
HEADER = """#pragma once
#include <cuda_runtime.h>
extern "C" long lowd_test_fail_at;
static inline cudaError_t lowd_test_alloc(void** p, size_t n, cudaMemPool_t pool, cudaStream_t s) {
    if (lowd_test_fail_at > 0 && --lowd_test_fail_at == 0) return cudaErrorMemoryAllocation;
    return cudaMallocFromPoolAsync(p, n, pool, s);
}
#define cudaMallocFromPoolAsync lowd_test_alloc
"""


def test_no_state_is_lost(tmp_path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2307_15969_gb300 import build
    build.build()
    (tmp_path / "fail.h").write_text(HEADER)
    (tmp_path / "fail.cu").write_text('extern "C" long lowd_test_fail_at;\nlong lowd_test_fail_at = 0;\n')
    nvcc = [build._nvcc()] + build.ARCH

    def compile_unit(src, obj, extra):
        p = subprocess.run(nvcc + build.NVCC_FLAGS + extra + ["-c", src, "-o", obj], capture_output=True, text=True)
        assert p.returncode == 0, p.stdout + p.stderr

    jobs = [(os.path.join(build.CSRC, u + ".cu"), str(tmp_path / (u + ".o")), ["-include", str(tmp_path / "fail.h")])
            for u in UNITS]
    jobs.append((str(tmp_path / "fail.cu"), str(tmp_path / "fail.o"), []))
    with cf.ThreadPoolExecutor(len(jobs)) as ex:
        list(ex.map(lambda j: compile_unit(*j), jobs))
    rest = [os.path.join(build.OBJ, f) for f in sorted(os.listdir(build.OBJ))
            if f.endswith(".o") and f[:-2] not in UNITS and os.path.exists(os.path.join(build.CSRC, f[:-2] + ".cu"))]
    lib = str(tmp_path / "liblowd.so")
    p = subprocess.run(nvcc + ["-shared", "-cudart", "static", "-o", lib] + [j[1] for j in jobs] + rest,
                       capture_output=True, text=True)
    assert p.returncode == 0, p.stdout + p.stderr
    p = subprocess.run([sys.executable, os.path.join(HERE, "_alloc_child.py"), lib], capture_output=True, text=True,
                       timeout=300)
    assert p.returncode == 0 and "ALLOC_OK" in p.stdout, p.stdout[-2000:] + p.stderr[-3000:]
