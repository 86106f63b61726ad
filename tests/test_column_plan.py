"""The grid of a one-launch Gram-Schmidt column leaves room for other contexts on short vectors: planned
here on the host, against a stand-in for the CUDA runtime with 152 SMs."""
import os
import shutil
import subprocess

import pytest

from test_device_limits import FAKE, ROOT

MAIN = r"""
template <class T> static void show(long long K) {
  const pcexp::ColumnPlan p = pcexp::plan_cgs_column<T>(K);
  std::printf("%d %lld %d %d\n", (int)sizeof(T), K, p.blocks, p.rows);
}
int main() {
  for (long long K : {64LL, 384LL, 6144LL, 27648LL, 38912LL, 38976LL, 110592LL, 1880064LL, 1958592LL}) show<double>(K);
  for (long long K : {64LL, 384LL, 6144LL, 27648LL, 110592LL, 214016LL, 214080LL, 1213504LL, 1259712LL}) show<float>(K);
  return 0;
}
"""


def test_short_vectors_leave_room_for_other_contexts(tmp_path):
    if shutil.which("nvcc") is None and not os.path.exists("/usr/local/cuda/bin/nvcc"):
        pytest.skip("no CUDA toolkit to build the library")
    from paper_1801_06300_gb300 import build
    build()
    pkg = os.path.join(ROOT, "paper_1801_06300_gb300")
    obj = os.path.join(pkg, "_build", "krylov_kernels.cu.o")
    if not os.path.exists(obj):
        pytest.skip("the library was built without its objects")
    src = tmp_path / "plan.cpp"
    src.write_text(FAKE.split("int main()")[0] + MAIN)
    exe = str(tmp_path / "plan")
    subprocess.run(["g++", "-std=c++17", "-O1", "-w", "-I/usr/local/cuda/include", "-I", os.path.join(pkg, "csrc"),
                    str(src), obj, "-o", exe, "-lpthread"], check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True, timeout=60).stdout.split("\n")[:-1]
    plans = [tuple(map(int, line.split())) for line in out]
    assert len(plans) == 18
    for size, K, blocks, rows in plans:
        limit = {8: 100 * 1024, 4: 32 * 1024}[size]
        if blocks == 0:  # the separate passes
            assert -(-K // 152) * size > limit - 64 * size
            continue
        assert blocks <= 152 and rows % 64 == 0 and rows * size <= limit
        assert (blocks - 1) * rows < K <= blocks * rows, "every block has rows"
        if K <= 6144 or (size == 4 and K <= 27648):  # four contexts at once, two blocks per SM
            assert 4 * blocks <= 2 * 152, (size, K, blocks)
