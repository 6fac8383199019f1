"""The chunk sizes the apply kernel takes, evaluated on the host by a small
program built against csrc/common.cuh. No kernels run."""
import subprocess

import pytest

from paper_2509_14433_gb300 import build as B


@pytest.mark.parametrize("V", [24577, 65536, 100003, 131072, 1 << 21])
def test_a_sparse_batch_has_a_chunk_for_every_warp(tmp_path, V):
    # most vertices get one or two records, which are not padded: the chunks
    # must not be sized for padding that is not there, or warps go without
    src, exe = tmp_path / "p.cu", tmp_path / "p"
    src.write_text(f"""#include <stdio.h>
#include "common.cuh"
using namespace cupc;
int main() {{
  unsigned bad = 0, seen = 0;
  for (uint32_t most : {{64u, 128u, 256u, 512u}})
    for (uint32_t warps : {{608u, 760u, 1013u}})
      for (uint64_t n = kSmallEdges + 1; 2 * n < 4ull * {V}u; n += n / 50 + 1) {{
        const uint32_t nrec = (uint32_t)(2 * n), c = chunk_records(nrec, {V}u, warps, most);
        if (nrec / warps < kStage) continue;
        seen++;
        bad += nrec / c < warps || c > most;
      }}
  printf("%u %d", bad, seen > 20);
}}
""")
    subprocess.run([B.NVCC, *B.ARCH, *B.FLAGS, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split() == ["0", "1"]


def test_long_chunks_only_where_one_or_two_a_warp_are_enough(tmp_path):
    src, exe = tmp_path / "p.cu", tmp_path / "p"
    src.write_text("""#include <stdio.h>
#include "common.cuh"
using namespace cupc;
int main() {
  unsigned bad = 0, longer = 0;
  for (uint32_t V : {2u, 300u, 2457u, 2458u, 8192u, 40000u, 1u << 21})
    for (uint32_t warps : {1u, 32u, 608u, 760u, 1013u})
      for (uint64_t n = 1; n < (1ull << 31) - 1; n = n * 21 / 20 + 1) {
        const uint32_t nrec = (uint32_t)(2 * n), most = default_most(nrec, V, warps);
        const uint32_t c = chunk_records(nrec, V, warps, most);
        bad += most != kDefaultItemRecords && most != kItemRecords;
        bad += c > kDefaultItemRecords && (nrec < 10ull * V || 2ull * c * warps < nrec);
        bad += c % kPad || c > most;
        longer += c > kDefaultItemRecords;
      }
  printf("%u %d", bad, longer > 100);
}
""")
    subprocess.run([B.NVCC, *B.ARCH, *B.FLAGS, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split() == ["0", "1"]
