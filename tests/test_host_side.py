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
