"""Kernels that read the stored face Jacobians as blocks are not compiled for the forms that store
16-value records instead (a block's index would run past a record's end)."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1801_06300_gb300", "csrc")


@pytest.mark.parametrize("scalar,dim,compiles", [("float", 3, False), ("double", 3, True)])
def test_transpose_from_blocks_refuses_records(tmp_path, scalar, dim, compiles):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no CUDA toolkit")
    src = tmp_path / "inst.cu"
    src.write_text(f"""#include "dg_kernels.cuh"
namespace pcexp {{
template cudaError_t jac_adjoint_p<{scalar}, {dim}, 1>(const DGData<{scalar}>&, LinData<{scalar}>, const {scalar}*,
                                                       {scalar}*, {scalar}*, const {scalar}*, {scalar}, cudaStream_t);
}}
""")
    r = subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-I", CSRC, "-c", str(src),
                        "-o", str(tmp_path / "inst.o")], capture_output=True, text=True)
    assert (r.returncode == 0) == compiles, r.stderr[-2000:]
    if not compiles:
        assert "not a record" in r.stderr
