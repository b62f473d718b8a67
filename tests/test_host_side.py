"""Host-side behaviour of the library that needs no GPU."""
import os
import subprocess
import sys

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
