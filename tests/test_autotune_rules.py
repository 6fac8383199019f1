"""What the autotuner times and keeps (no GPU): only batch sizes that reach
the tuned kernel, and only settings that beat the default by more than runs
differ."""
import json
import subprocess

import pytest

from paper_2509_14433_gb300 import autotune as AT
from paper_2509_14433_gb300 import build as B


def test_small_batches_are_the_library_s(tmp_path):
    src, exe = tmp_path / "p.cu", tmp_path / "p"
    src.write_text('#include <stdio.h>\n#include "common.cuh"\nint main() { printf("%u", cupc::kSmallEdges); }\n')
    subprocess.run([B.NVCC, *B.ARCH, *B.FLAGS, str(src), "-o", str(exe)], check=True)
    assert int(subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout) == AT.SMALL_EDGES


@pytest.mark.parametrize("most", [1 << 14, 1 << 18, 1 << 22])
def test_sizes_reach_the_tuned_kernel(most):
    sizes = AT.default_sizes(most)
    assert all(AT.SMALL_EDGES < n <= most for n in sizes)
    buckets = [AT.bucket_of(n) for n in sizes]
    assert buckets == list(range(AT.bucket_of(AT.SMALL_EDGES), AT.bucket_of(most) + 1))


def test_a_setting_is_kept_only_beyond_the_noise():
    default, other = (256, 8, 0), (64, 8, 0)
    assert AT.choose(other, [1.0, 1.1], default, [1.2, 1.3])[0] == other
    assert AT.choose(other, [1.0, 1.2], default, [1.15, 1.3])[0] == default
    assert AT.choose(default, [1.0, 1.2], default, [1.0, 1.2]) == (default, 1.1)


def test_table_holds_no_setting_of_a_size_that_is_not_tuned():
    with open(AT.DEFAULT_CACHE) as f:
        table = json.load(f)
    for shapes in table.values():
        for entries in shapes.values():
            for bucket, e in entries.items():
                assert e["edges"] > AT.SMALL_EDGES and AT.bucket_of(e["edges"]) == int(bucket)
