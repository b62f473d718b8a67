"""Host-side behaviour of the library that needs no GPU."""
import os
import subprocess
import sys

import pytest

import paper_1409_5705_b200 as S

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_workspace_bytes_makes_no_cuda_call():
    """sfb_workspace_bytes is host-only: a program may ask it before it forks the processes that use the GPU.  The first CUDA call of a
    process looks for the driver's library, which the loader's own trace shows."""
    prog = """
import ctypes, paper_1409_5705_b200 as S
for model in (S.MLR, S.DML, S.SC, S.L2MLR):
    for prec in (S.PREC_BF16, S.PREC_FP32, S.PREC_FP32_FFMA):
        for shape in ((4999, 3004, 7, 37), (2000, 1000, 8, 16), (10000, 20000, 16, 64), (300, 200, 1, 8)):
            for nnz in (0, 5000):
                S.sfb_workspace_bytes(S.make_config(model, *shape, 0.1, prec, sdca_lambda=0.1, sdca_n=10, csr_nnz_max=nnz))
print("asked")
"""
    out = subprocess.run([sys.executable, "-c", prog], cwd=ROOT, env=dict(os.environ, LD_DEBUG="libs"), capture_output=True, text=True)
    assert out.returncode == 0 and "asked" in out.stdout, out.stderr[-500:]
    assert "libcuda.so" not in out.stderr


@pytest.mark.parametrize("model,rows,cols,K", [(S.MLR, 1_100_000, 20_000, 64), (S.DML, 200_000, 110_000, 64), (S.SC, 1_000_000, 20_000, 8),
                                               (S.SC, 700_000, 20_000, 64), (S.L2MLR, 2_000_000, 11_000, 100)])
def test_fp32_contexts_fit_the_gpu_where_w_does(model, rows, cols, K):
    """The pairs of W that the fp32 mode derives must not be what keeps a matrix from fitting the 180 GB."""
    kw = dict(sdca_lambda=0.1, sdca_n=1) if model == S.L2MLR else {}
    assert 4 * rows * cols + S.sfb_workspace_bytes(S.make_config(model, rows, cols, 1, K, 0.1, S.PREC_FP32, **kw)) <= 165e9
    # (and are still derived where they fit)
    assert S.sfb_workspace_bytes(S.make_config(model, rows // 4, cols, 1, 200, 0.1, S.PREC_FP32, **kw)) >= rows * cols


# csrc/sfb_api.cu against a fake of the CUDA runtime that counts the copies in flight: the n-th fallible call fails.
FAKE = r"""
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
static std::map<void*, int> in_flight;      // host copies enqueued per stream
static int calls = 0, fail_at = -1, step_rc = 0, host_parts = 4;
static bool joined = false;
static bool failing() { return calls++ == fail_at; }
#include "sfb_api.cu"
extern "C" {
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = reinterpret_cast<cudaStream_t>(2); return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { *e = reinterpret_cast<cudaEvent_t>(1); return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { *p = calloc(1, n); return cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { free(p); return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return failing() ? cudaErrorUnknown : cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return failing() ? cudaErrorUnknown : cudaSuccess; }
cudaError_t cudaMemcpyAsync(void*, const void*, size_t, cudaMemcpyKind k, cudaStream_t s) {
  if (failing()) return cudaErrorUnknown;
  if (k == cudaMemcpyHostToDevice) in_flight[s]++;
  return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
  in_flight[s] = 0;
  if (joined && s == reinterpret_cast<cudaStream_t>(1)) in_flight[reinterpret_cast<cudaStream_t>(2)] = 0;
  return cudaSuccess;
}
}
namespace sfb {
int tc_host_parts(const sfb_ctx*) { return host_parts; }
int tc_factors(sfb_ctx*, int64_t, int64_t, const float*, const float*, const int32_t*, bool, float*) {
  joined = step_rc == 0;                    // the step's stream has waited for the copies' events
  return step_rc;
}
int tc_update(sfb_ctx*) { return SFB_OK; }
void tc_destroy(sfb_ctx*) {}
}
int main() {
  for (int parts : {4, 1})
    for (step_rc = 0; step_rc >= -1; --step_rc)
      for (fail_at = -1; fail_at < 24; ++fail_at) {
        sfb_ctx* ctx = new sfb_ctx();
        ctx->cfg.model = SFB_MLR; ctx->cfg.precision = SFB_PREC_BF16;
        ctx->cfg.rows = 8; ctx->cfg.cols = 8; ctx->cfg.workers = 1; ctx->cfg.batch = 512;
        ctx->K = 512; ctx->in_dim = 8;
        alignas(1024) static char ws[1 << 16];
        ctx->ws = ws;
        ctx->lay.loss = 4096; ctx->lay.scalars = 1024; ctx->lay.stageX = 8192; ctx->lay.stageL = 32768;
        ctx->stream = reinterpret_cast<cudaStream_t>(1);
        calls = 0;
        joined = false;
        host_parts = parts;
        in_flight.clear();
        alignas(16) static float X[512 * 8];
        static int32_t y[512];
        float loss;
        uint32_t status;
        const int rc = sfb_step_host(ctx, X, nullptr, y, &loss, &status);
        for (auto& f : in_flight)
          if (f.second) { printf("rc %d with %d copies in flight (call %d failed, step %d)\n", rc, f.second, fail_at, step_rc); return 1; }
        if (ctx->host && ctx->host->parts) { printf("parts left set\n"); return 1; }
        if ((rc != 0) != (step_rc != 0 || (fail_at >= 0 && fail_at < calls))) { printf("rc %d, call %d\n", rc, fail_at); return 1; }
        sfb_destroy(ctx);
      }
  printf("ok\n");
  return 0;
}
"""


def test_host_step_returns_no_buffer_that_is_still_read(tmp_path):
    src, exe = tmp_path / "fake.cpp", tmp_path / "fake"
    src.write_text(FAKE)
    csrc = os.path.join(ROOT, "paper_1409_5705_b200", "csrc")
    cuda = next(p for p in ("/usr/local/cuda", "/usr/local/cuda-12.9") if os.path.exists(os.path.join(p, "include", "cuda_runtime.h")))
    subprocess.check_call(["g++", "-std=c++17", "-w", "-I", os.path.join(ROOT, "include"), "-I", csrc, "-I", os.path.join(cuda, "include"), str(src),
                           "-o", str(exe), "-Wl,--unresolved-symbols=ignore-all"])
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout + out.stderr


def test_kernels_read_nothing_before_their_wait():
    """A kernel launched ahead of the one before it waits for that one.  Its `__restrict__` parameters all go through the wait: the compiler
    may move accesses through the others above it."""
    import glob
    import re
    seen = 0
    for path in glob.glob(os.path.join(ROOT, "paper_1409_5705_b200", "csrc", "*.cu")):
        src = open(path).read()
        for m in re.finditer(r"__global__[^;{]*?\(((?:[^(){}]|\([^()]*\))*)\)\s*\{", src):
            names = re.findall(r"__restrict__\s+(\w+)", m.group(0))
            if names:
                wait = re.search(r"pdl_wait\(([^)]*)\);", src[m.end():])
                assert wait and sorted(names) == sorted(wait.group(1).replace(" ", "").split(",")), (os.path.basename(path), m.group(0)[:120])
                seen += 1
    assert seen >= 30
