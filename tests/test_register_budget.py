"""The register count of the sweep that reads its M from the tensor cores' buffer (order 6, FP32): at most
64, so that eight blocks of four warps stay on an SM.  An address kept for the forms of M that this
sweep does not use is enough to lose the eighth block, and a fifth of its speed on a full GPU.  And the
checkpointing adjoint of order 5, which has no register to spare at its five blocks: no spills.  Compiles the
one kernel and reads what the assembler prints.
"""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"

pytestmark = pytest.mark.skipif(not os.path.exists(NVCC), reason="no nvcc")


def _assemble(tmp_path, header, kernel):
    src = tmp_path / "one.cu"
    csrc = os.path.join(ROOT, "paper_2502_08470_gb300", "csrc")
    src.write_text(f'#include "{csrc}/{header}"\n'
                   f"namespace sk {{ const void* one() {{ return reinterpret_cast<const void*>(&{kernel}); }} }}\n")
    r = subprocess.run([NVCC, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-rdc=true", "-lineinfo",
                        "-Xptxas", "-v", "-c", str(src), "-o", str(tmp_path / "one.o")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    used = [int(m) for m in re.findall(r"Used (\d+) registers", r.stderr)]
    assert len(used) == 1, r.stderr
    return used[0], sum(int(m) for m in re.findall(r"(\d+) bytes spill", r.stderr))


def test_precomputed_m_sweep_fits_eight_blocks(tmp_path):
    used, spills = _assemble(tmp_path, "sk_fwd_poly.cuh", "fwd_poly_kernel<float, 6, 6, false, false, false, true>")
    assert used <= 64 and spills == 0


def test_checkpointing_adjoint_does_not_spill(tmp_path):
    used, spills = _assemble(tmp_path, "sk_bwd_poly.cuh", "bwd_approx_kernel<float, 5, 4, 8>")
    assert used <= 96 and spills == 0
