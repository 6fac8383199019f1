"""Host rules of the native code at the edges of what its entry points accept,
evaluated by small programs built against csrc/common.cuh. No kernels run."""
import subprocess

import pytest

from paper_2509_14433_gb300 import build as B


def _run(tmp_path, body):
    """The output of a program with `body` as its main function."""
    src, exe = tmp_path / "p.cu", tmp_path / "p"
    src.write_text('#include <stdio.h>\n#include "common.cuh"\nusing namespace cupc;\nint main() {\n' + body + "\nreturn 0;\n}\n")
    res = subprocess.run([B.NVCC, *B.ARCH, *B.FLAGS, str(src), "-o", str(exe)], capture_output=True, text=True)
    assert res.returncode == 0, res.stderr
    res = subprocess.run([str(exe)], capture_output=True, text=True)
    assert res.returncode == 0, res.stderr
    return res.stdout


@pytest.mark.parametrize("V", [2, 700, 3000, 16384, 131072, 1 << 21])
def test_every_accepted_setting_gives_chunks_of_whole_groups(tmp_path, V):
    # a vertex's padded records start at multiples of kPad, and the apply
    # kernel takes them kPad at a time: no chunk may split a group
    out = _run(tmp_path, f"""
  const uint32_t V = {V}u;
  unsigned long long bad = 0, most_used = 0;
  for (uint32_t most = kMinItemRecords; most <= kItemRecords; most++)
    for (uint32_t warps : {{1u, 3u, 32u, 152u, 608u, 760u, 1013u, 3040u}})
      for (uint64_t n = 1; n < (1ull << 31) - 1; n = n * 3 / 2 + 1) {{
        const uint32_t c = chunk_records((uint32_t)(2 * n), V, warps, most);
        bad += c == 0 || c % kPad || c > most;
        most_used += c + kPad > most;
      }}
  printf("%llu %d", bad, most_used > 1000);""")
    assert out.split() == ["0", "1"]
