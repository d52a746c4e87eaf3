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


def test_trip_limit_of_the_collision_loops(tmp_path):
    """The limit leaves room for every step that ends: with mean dt nu_max, an
    electron's draws exceed it by twelve standard deviations and 100 more with a
    probability below 1e-30 (float64: eight trips a draw of a pool; float32: the
    2^24 draws that its time left can count); and it is an int for any dt."""
    means = [0.0, 1e-3, 1.0, 20.0, 1e3, 1e5, 1e6, 1e7, 1.6e7, 1e8, 1e300]
    body = "".join(f'printf("%d %d\\n", kTripsF32, trip_limit(1e-12, {m} * 1e12));' for m in means)
    for m, (f32, f64) in zip(means, _run(tmp_path, body)):
        draws = m + 12 * m ** 0.5 + 100
        assert 2 ** 24 < int(f32) <= 2 ** 25 and int(f64) >= min(8 * draws, 2 ** 31 - 1), m


def test_error_flags_are_bits_of_their_own(tmp_path):
    """Each error that a kernel raises has a bit to itself, the draw limit's
    among them, and the context's message names every bit it can report."""
    rows = _run(tmp_path, "".join(f'printf("{n} %u\\n", (unsigned){n});' for n in (
        "kErrOutCapacity", "kErrChildCapacity", "kErrOverflow", "kErrStack", "kErrSplitCapacity", "kErrPhotoCapacity",
        "kErrPoissonLimit", "kErrBarrier", "kErrDraws")))
    bits = {n: int(v) for n, v in rows}
    assert all(v and v & (v - 1) == 0 for v in bits.values()) and len(set(bits.values())) == len(bits)
    text = open(os.path.join(B.CSRC, "pic.cu")).read().split("static int check_err")[1].split("\n}")[0]
    for n, v in bits.items():
        assert n == "kErrBarrier" or f"{v} " in text, n  # (a barrier only in batched swarms)


def test_float64_solves_keep_their_array_at_every_size():
    """The workspace that the binding allocates for a float64 solve grows with
    the cells alone: between boxes of 48^3 to 128^3 its bytes a cell differ by
    what is not proportional to them (partial sums, tables, padding), below 3 %;
    an array left out would be 19 %."""
    B.build()
    from paper_2110_14494_gb300 import picmcc as P
    per = {n: P._poisson_bytes(P.poisson_config(n, n, n, 1e-5, 0.0, 1.0, 1.0, 64)) / n ** 3 for n in range(48, 136, 8)}
    small = [v for n, v in per.items() if n > 88]  # above 32 MiB nothing is added to what the library states
    assert max(small) / min(small) < 1.03, per
    for n, v in per.items():
        assert v >= 0.97 * min(small), (n, v)
