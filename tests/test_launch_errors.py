"""Launch errors seen by the host code, against fakes of the CUDA runtime calls (CPU only): a small program that
defines the calls itself and loads libamgeig.so, whose references then bind to the fakes."""
import shutil
import subprocess
from pathlib import Path

import pytest

ROOT = Path(__file__).resolve().parents[1]

FAKES = r"""
#include <cuda_runtime_api.h>
#include <dlfcn.h>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include "kernels.cuh"

static cudaError_t pending = cudaSuccess;      // the thread's last error
static dim3 grid, block;                       // of the launch being made
static bool refuse_rows = false, no_cluster = false;
static float last_ms = 1.f;
static int rows = 0;

extern "C" {
cudaError_t cudaGetLastError(void) { cudaError_t e = pending; pending = cudaSuccess; return e; }
cudaError_t cudaPeekAtLastError(void) { return pending; }
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void*, const cudaLaunchConfig_t*) {
  *n = 0;
  if (!no_cluster) { *n = 1; return cudaSuccess; }
  return pending = cudaErrorInvalidClusterSize;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t*, const void*, void**) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = (cudaEvent_t)1; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = last_ms; return cudaSuccess; }
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t, struct CUstream_st*) { grid = g; block = b; return 0; }
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* s, void* st) {
  *g = grid; *b = block; *s = 0; *(void**)st = nullptr; return cudaSuccess;
}
cudaError_t __cudaGetKernel(void** k, const void* f) { *k = (void*)f; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(void*, dim3 g, dim3, void**, size_t, cudaStream_t) {
  const bool by_row = (int)g.x == rows;        // one block per row
  last_ms = by_row ? 0.001f : 1.f;             // a refused launch takes no time
  if (by_row && refuse_rows) return pending = cudaErrorInvalidConfiguration;
  return cudaSuccess;
}
}

using namespace amgeig;

int main(int argc, char** argv) {
  void* lib = dlopen(argv[1], RTLD_NOW);
  if (!lib) { std::printf("%s\n", dlerror()); return 2; }
  const char* what = argv[2];
  if (!std::strncmp(what, "tune", 4)) {
    auto tune = (TuneResult(*)(DevCsr&, int, int, const float*, const float*, const float*, float*, cudaStream_t))
        dlsym(lib, "_ZN6amgeig11autotune_f4ERNS_6DevCsrEiiPKfS3_S3_PfP11CUstream_st");
    refuse_rows = !std::strcmp(what, "tune-refused");
    rows = 1000;
    DevCsr S;
    S.rows = S.cols = rows;
    S.nnz = 40 * rows;
    const int w4 = std::atoi(argv[3]);
    tune(S, 0, w4, nullptr, nullptr, nullptr, nullptr, nullptr);
    std::printf("%d\n", S.tuned[w4]);
  } else {
    const bool entry = !std::strcmp(what, "fits-entry");
    std::vector<char> work(4096, 0);
    PencilWork* w = (PencilWork*)work.data();
    no_cluster = true;
    pending = std::atoi(argv[3]) ? cudaErrorInvalidValue : cudaSuccess;
    if (entry) {
      auto f = (void (*)(PencilWork*, int, int, const double*, double*, double*, cudaStream_t))
          dlsym(lib, "_ZN6amgeig11launch_eighEPNS_10PencilWorkEiiPKdPdS4_P11CUstream_st");
      f(w, 400, 8, nullptr, nullptr, nullptr, nullptr);
    } else {
      auto f = (void (*)(PencilWork*, int, int, const double*, double*, double*, cudaStream_t, const int*))
          dlsym(lib, "_ZN6amgeig14launch_syev_dfEPNS_10PencilWorkEiiPKdPdS4_P11CUstream_stPKi");
      f(w, 400, 8, nullptr, nullptr, nullptr, nullptr, nullptr);
    }
    std::printf("%d\n", cudaPeekAtLastError() != cudaSuccess);
  }
  return 0;
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    from paper_1503_08462_gb300 import _build

    lib = _build.build_cuda_lib()
    nvcc = shutil.which("nvcc")
    include = Path(nvcc).resolve().parents[1] / "include"
    if not (include / "cuda_runtime_api.h").exists():
        pytest.skip("no CUDA headers beside nvcc")
    d = tmp_path_factory.mktemp("fakes")
    (d / "fakes.cpp").write_text("#include <vector>\n" + FAKES)
    subprocess.run(["g++", "-std=c++17", "-rdynamic", "-I", str(include), "-I", str(_build.CUDA_DIR),
                    str(d / "fakes.cpp"), "-o", str(d / "fakes"), "-ldl"], check=True)

    def call(*args):
        r = subprocess.run([str(d / "fakes"), str(lib), *map(str, args)], capture_output=True, text=True, timeout=120)
        assert r.returncode == 0, r.stdout + r.stderr
        return int(r.stdout)

    return call


@pytest.mark.parametrize("w4", [1, 5, 8, 9, 16, 17, 20, 32])
def test_refused_tuning_launch_leaves_the_rule(run, w4):
    """A block-per-row trial whose launch is refused looks fastest (it takes no time); the operator must stay
    untuned, as its shape does not fit the encoding of the others."""
    assert run("tune-refused", w4) == 0
    assert run("tune", w4) == 128  # the same trial, launched: chosen


@pytest.mark.parametrize("solver", ["fits", "fits-entry"])
def test_cluster_query_keeps_an_earlier_error(run, solver):
    """Asking whether a cluster can be resident (the answer is no, as an error) must not clear the error of an
    earlier launch, and leaves none of its own."""
    assert run(solver, 1) == 1
    assert run(solver, 0) == 0
