"""The kernels' bounds arithmetic (csrc/bounds.h), compiled and run on the host."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2205_06327_gb300", "csrc")


def _run(tmp_path, body: str) -> list[int]:
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    src = tmp_path / "t.cpp"
    src.write_text('#include <cstdio>\n#include "bounds.h"\nusing namespace ptycho;\nint main() {\n' + body + "}\n")
    subprocess.run([cxx, "-std=c++17", "-I", CSRC, str(src), "-o", str(tmp_path / "t")], check=True)
    out = subprocess.run([str(tmp_path / "t")], check=True, capture_output=True, text=True).stdout
    return [int(v) for v in out.split()]


@pytest.mark.parametrize("M,W", [(4096, 524416), (4096, 524417), (1024, 2100000), (8, 2**31 - 1), (1024, 2**24)])
def test_window_offsets_of_wide_objects(tmp_path, M, W):
    """The last element of a window in the widest objects a plan accepts (2^34 pixels) is reached."""
    assert M * W <= 2**34
    at = _run(tmp_path, f'std::printf("%lld %lld\\n", (long long)window_at({M - 1}, {M - 1}, {W}), '
                        f'(long long)window_at({M - 1}, 0, {W}));')
    assert at == [(M - 1) * W + M - 1, (M - 1) * W]


@pytest.mark.parametrize("blocks", [1, 2, 4, 8])
@pytest.mark.parametrize("need", [1000, 38000, 60000])
def test_shared_memory_limits_the_resident_blocks(tmp_path, blocks, need):
    """One block more than the limit does not fit on an SM; the limit itself fits
    unless the kernel's own need is larger.  The cluster chain's limit is what
    tensor memory serves."""
    smem, cols, sm, block = _run(tmp_path, f'std::printf("%zu %d %zu %zu\\n", smem_for_at_most({blocks}, {need}), '
                                           'kTmemColumns, kSmShared, kBlockShared);')
    assert smem >= need and smem % 128 in (0, need % 128) and (blocks + 1) * (smem + block) > sm
    assert smem == need or blocks * (smem + block) <= sm
    assert cols // 128 == 4
