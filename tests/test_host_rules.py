"""Host-side rules of the CUDA sources, compiled from the headers that the
kernels and their launches use and run without a GPU."""
import os
import subprocess

import pytest

from paper_2110_14494_gb300 import build as B


def _run(tmp_path, body):
    try:
        nvcc = B._nvcc()
    except RuntimeError as e:
        pytest.skip(str(e))
    src, exe = tmp_path / "rules.cu", tmp_path / "rules"
    src.write_text('#include <stdio.h>\n#include "common.cuh"\nusing namespace pic;\nint main() {\n' + body + "\nreturn 0; }\n")
    subprocess.check_call([nvcc, *B.ARCH, "-std=c++17", "-I", B.CSRC, str(src), "-o", str(exe)])
    return [line.split() for line in subprocess.check_output([str(exe)]).decode().splitlines()]


def test_tables_of_a_batch_begin_on_16_bytes(tmp_path):
    """Every length that a gas table may have (2 to 4096 nodes): one table holds
    its ten reals a node, and the next begins on a multiple of 16 bytes in
    either precision, as the 16-byte loads of its rows need."""
    rows = _run(tmp_path, 'for (int n = 2; n <= 4096; ++n) printf("%d %zu\\n", n, table_reals(n));')
    assert [int(n) for n, _ in rows] == list(range(2, 4097))
    for n, reals in ((int(a), int(b)) for a, b in rows):
        assert 10 * n <= reals <= 10 * n + 3, n
        assert reals * 4 % 16 == 0, n
    # the binary that runs lays its batches out by that rule
    used = "".join(open(os.path.join(B.CSRC, f)).read() for f in ("pic.cu", "swarm_batch.cuh"))
    assert "kTableStride" not in used
