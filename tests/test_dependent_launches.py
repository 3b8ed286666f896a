"""Host checks of how kernels are launched: behind one another (csrc/pdl.cuh), and with
more shared memory than by default.  The runtime's calls are replaced by fakes."""
import glob
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1609_01490_gb300", "csrc")


def test_no_read_only_loads_behind_a_producer():
    """Files whose kernels are launched behind another use no load that takes its data
    as constant for the whole kernel: the first kernel may still be writing it."""
    files = [f for f in glob.glob(os.path.join(CSRC, "*.cu")) if "launch_behind" in open(f).read()]
    assert len(files) >= 4
    for f in files:
        code = re.sub(r"//[^\n]*", "", open(f).read())
        assert not re.search(r"__ldg\s*\(|ld\.global\.nc", code), f


def _run(tmp_path, *sources):
    """Exit status of a program made of the given sources; what they define stands in
    front of the CUDA runtime's own calls."""
    nvcc = next((c for c in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", shutil.which("nvcc"))
                 if c and os.path.exists(c)), None)
    if nvcc is None:
        pytest.skip("no nvcc")
    exe = str(tmp_path / "launch")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-cudart", "shared", "-I", CSRC,
                    "-o", exe, *(str(s) for s in sources)], check=True)
    lib = os.path.join(os.path.dirname(os.path.dirname(nvcc)), "lib64")
    env = dict(os.environ, LD_LIBRARY_PATH=os.pathsep.join([lib, os.environ.get("LD_LIBRARY_PATH", "")]))
    return subprocess.run([exe], env=env).returncode


def test_failed_launch_leaves_no_error(tmp_path):
    """A launch that fails reports its error and leaves none for the next call that asks
    the runtime for the last one."""
    (tmp_path / "launch.cu").write_text('''#include "pdl.cuh"
#include "tri_internal.h"
extern "C" int last_error;
__global__ void nothing(int *p) { (void)p; }
int main()
{
    const cudaError_t e = trihost::launch_behind(nothing, dim3(1), dim3(32), 0, nullptr, (int *)nullptr);
    if (e != cudaErrorInvalidConfiguration || last_error != 0) return 1;
    const cudaError_t a = trihost::allow_smem(nothing, 1024);
    return a == cudaErrorInvalidValue && last_error == 0 ? 0 : 2;
}
''')
    # in front of the runtime's own: both calls fail and leave their error behind
    (tmp_path / "fakes.cpp").write_text('''extern "C" {
int last_error = 0;
int cudaLaunchKernelExC(const void *, const void *, void **) { return last_error = 9; }
int cudaFuncSetAttribute(const void *, int, int) { return last_error = 1; }
int cudaGetLastError()
{
    const int e = last_error;
    last_error = 0;
    return e;
}
}
''')
    assert _run(tmp_path, tmp_path / "launch.cu", tmp_path / "fakes.cpp") == 0


def test_shared_memory_limit_is_one_value(tmp_path):
    """The limit of a kernel's shared memory belongs to the process: calls of different
    sizes all set the same one, so that none lowers it between another thread's call
    and launch, and it covers every launch."""
    (tmp_path / "main.cu").write_text('''#include "../../include/tri.h"
extern "C" int bad;
int main()
{
    float *f = (float *)4096;
    size_t bytes = 0;
    const uint32_t shapes[][4] = {{8, 64, 128, 128}, {8, 14, 128, 96}, {8, 14, 64, 64}, {100000, 14, 128, 128},
                                  {100000, 64, 8, 5}, {100000, 64, 32, 64}, {5000, 64, 128, 1}, {100000, 64, 1, 1}};
    for (const auto &s : shapes) {
        tri_mlp_workspace_size(s[0], s[2], s[3], &bytes);
        if (tri_mlp_forward(f, f, s[0], s[1], s[2], s[3], f, f, bytes, nullptr) != TRI_OK) return 1;
        if (tri_mlp_grad(f, f, f, s[0], s[1], s[2], s[3], f, f, f, bytes, nullptr) != TRI_OK) return 2;
    }
    const uint32_t counts[] = {1, 10, 4095, 4096, 100000};
    for (uint32_t count : counts)
        for (uint32_t d : {3u, 64u})
            for (uint32_t reg : {1u, 4u, 8u}) {
                tri_edm_batched_workspace_size(count, &bytes);
                if (tri_edm_batched(f, (uint64_t *)f, (uint32_t *)f, count, d, f, (uint64_t *)f, 16, reg, f, bytes,
                                    nullptr) != TRI_OK)
                    return 3;
            }
    return bad;
}
'''.replace("../../include/tri.h", os.path.join(ROOT, "include", "tri.h")))
    (tmp_path / "fakes.cpp").write_text('''#include <cstddef>
#include <map>
struct dim3 { unsigned x, y, z; };
struct Config { dim3 grid, block; size_t smem; };
static std::map<const void *, int> limit;
extern "C" {
int bad = 0;
static int launch(const void *f, size_t smem)
{
    const auto l = limit.find(f);
    if (smem > 48 * 1024 && (l == limit.end() || smem > (size_t)l->second)) bad = 11;
    return 0;
}
int cudaFuncSetAttribute(const void *f, int, int v)
{
    const auto l = limit.emplace(f, v).first;
    if (l->second != v || v > 227 * 1024) bad = 10;
    return 0;
}
int cudaLaunchKernel(const void *f, dim3, dim3, void **, size_t smem, void *) { return launch(f, smem); }
int cudaLaunchKernelExC(const Config *c, const void *f, void **) { return launch(f, c->smem); }
int cudaGetLastError() { return 0; }
int cudaMemsetAsync(void *, int, size_t, void *) { return 0; }
int cudaGetDevice(int *d) { *d = 0; return 0; }
int cudaDeviceGetAttribute(int *v, int, int) { *v = 152; return 0; }
int cudaOccupancyMaxActiveBlocksPerMultiprocessor(int *n, const void *, int, size_t) { *n = 2; return 0; }
int cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *, int, size_t, unsigned) { *n = 2; return 0; }
}
''')
    assert _run(tmp_path, tmp_path / "main.cu", tmp_path / "fakes.cpp", os.path.join(CSRC, "mlp.cu"),
                os.path.join(CSRC, "edm_batched.cu")) == 0
