"""The shared-memory layout of the canonical SMEM sweep, evaluated on the host: no array overlaps another one
that is live with it, in any mode and at any side that the layout serves."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2511_20911_gb300", "csrc")
REC, PLAIN, PACKED = 0, 1, 2


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path_factory.mktemp("layout") / "smem_layout_host")
    subprocess.check_call([nvcc, "-O1", "-std=c++17", "-I", CSRC, "-o", exe, os.path.join(HERE, "smem_layout_host.cu")])
    return exe


@pytest.fixture(scope="module")
def layouts(exe):
    """(L, Lc, paper, n_seg, mode) -> {array: (first word, end)} over every segment cut of the sides."""
    sides = [(L, L) for L in range(4, 98, 2)] + [(4, 64), (64, 4), (6, 96), (18, 96), (96, 18), (38, 52)]
    cases = [(L, Lc, paper, n_seg, mode) for L, Lc in sides for paper in (0, 1) for mode in (REC, PLAIN, PACKED)
             for n_seg in sorted({-(-(Lc // 2) // 3), -(-(Lc // 2) // 2), Lc // 2})]
    out = subprocess.run([exe], input="".join("%d %d %d %d %d\n" % c for c in cases), capture_output=True, text=True,
                         check=True)
    lines = [ln.split() for ln in out.stdout.strip().split("\n")]
    assert len(lines) == len(cases)
    return {c: {ln[k]: (int(ln[k + 1]), int(ln[k + 2])) for k in range(0, len(ln), 3)} for c, ln in zip(cases, lines)}


def overlap(a, b):
    return a[0] < b[1] and b[0] < a[1]


def test_arrays_are_disjoint(layouts):
    for case, arrays in layouts.items():
        items = [(n, r) for n, r in arrays.items() if n != "total" and r[1] > r[0]]
        for k, (n, r) in enumerate(items):
            assert 260 <= r[0] and r[1] <= arrays["total"][1], (case, n)
            for m, q in items[:k]:
                assert not overlap(r, q), (case, n, m)


def test_correlation_scratch_stays_in_the_dead_hidden_words(layouts):
    """A correlation sample (square lattices) writes its scratch over the hidden words: a word per row and chain
    up to L = 32, a word per site beyond.  Rows, records, expansion table and tables are live then."""
    for (L, Lc, paper, n_seg, mode), arrays in layouts.items():
        if L != Lc:
            continue
        scratch = (arrays["w"][0], arrays["w"][0] + (32 * L if L <= 32 else L * L))
        for n in ("rows", "rec", "expand", "tab"):
            if arrays[n][1] > arrays[n][0]:
                assert not overlap(scratch, arrays[n]), (L, paper, n_seg, mode, n)
        assert scratch[1] <= arrays["total"][1], (L, paper, n_seg, mode)


@pytest.mark.parametrize("reserved,static,ok", [(1024, 0, 1), (1024, 4, 0), (1024, 128, 0), (0, 0, 0), (2048, 0, 0), (1020, 4, 0)])
def test_launchers_refuse_tables_at_another_address(exe, reserved, static, ok):
    """The row-form kernels return without work when their tables are not at shared address 16384: what the
    launchers ask before a launch covers the driver's reserved bytes and the kernel's static shared memory."""
    out = subprocess.run([exe, str(reserved), str(static)], capture_output=True, text=True, check=True)
    assert int(out.stdout) == ok


def test_no_static_shared_memory_in_the_row_form_kernels():
    """Static shared memory in a file of theirs would move the dynamic one (extern declarations are that)."""
    files = ["crbm_canon.cu", "crbm_canon_body.cuh", "crbm_row_core.cuh", "crbm_device.cuh", "crbm_generic_body.cuh",
             "crbm_bitplane_body.cuh", "crbm_bitplane_core.cuh", "crbm_batch_kernel.cuh", "crbm_batch.cu", "crbm_batch_small.cu"]
    for f in files:
        with open(os.path.join(CSRC, f)) as fh:
            for n, line in enumerate(fh, 1):
                code = line.split("//")[0]
                assert "__shared__" not in code or "extern __shared__" in code, f"{f}:{n}"
