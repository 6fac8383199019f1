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
        const uint32_t h = hub_chunk_records((uint32_t)(2 * n), warps, most);
        bad += c == 0 || c % kPad || c > most || h == 0 || h % kPad || h > most;
        most_used += c + kPad > most;
      }}
  printf("%llu %d", bad, most_used > 1000);""")
    assert out.split() == ["0", "1"]


def test_staging_holds_as_much_as_max_batch_says():
    # host batches and host pairs are staged max_batch at a time in two slots
    # of 8 bytes an edge and 1 an op, up to the largest max_batch there is
    from paper_2509_14433_gb300 import cupc as C
    top, less = (1 << 31) - 1, (1 << 31) - (1 << 23)
    for V in (2, 1000, 1 << 21):
        rows = 8 if V > 1000 else 0
        size = {B: C.cupc_workspace_bytes(V, (0, 0, rows, B)) for B in (less, top)}
        assert size[top] - size[less] >= 2 * 9 * (top - less) - 4 * 256
        assert C.cupc_workspace_bytes(V, (0, 0, rows, top + 1)) == 0


def test_record_offsets_of_the_longest_chunk_fit_32_bits(tmp_path):
    out = _run(tmp_path, """
  int ok = 1;
  for (uint64_t B = 1; B < (1ull << 31); B = B * 2 + 1)
    for (uint64_t V = 2; V <= kMaxVertices; V *= 2) {
      const uint32_t n = chunk_edges((uint32_t)B);
      ok &= n > 0 && n <= B && (n == B || n == kMaxChunkEdges) && rec_entries(V, n) < 0xFFFFFFFFull - 4096;
    }
  printf("%d", ok);""")
    assert out == "1"


def test_which_memory_a_kernel_stores_the_forest_to(tmp_path):
    # only the graph's own device's memory, aligned; the default attributes
    # (unregistered) are those of plain host memory and of a null pointer
    out = _run(tmp_path, """
  const cudaMemoryType types[4] = {cudaMemoryTypeUnregistered, cudaMemoryTypeHost, cudaMemoryTypeDevice,
                                   cudaMemoryTypeManaged};
  for (int t = 0; t < 4; t++)
    for (int dev = 0; dev < 2; dev++)
      for (uintptr_t off : {0, 4, 8}) {
        cudaPointerAttributes at{};
        at.type = types[t];
        at.device = dev;
        printf("%d", stores_directly(at, (void*)(0x1000 + off), 1));
      }
  printf(" %d", stores_directly(cudaPointerAttributes{}, nullptr, 0));""")
    assert out == "000000" * 2 + "000101" * 2 + " 0"
