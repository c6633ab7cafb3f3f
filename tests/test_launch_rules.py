"""Launch rules by sizes (crbm_launch.h), evaluated on the host for a GPU of 152 SMs: what they choose at sizes where
the variants were timed and another choice was found slower."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2511_20911_gb300", "csrc")


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path_factory.mktemp("rules") / "launch_rules_host")
    subprocess.check_call([nvcc, "-O1", "-std=c++17", "-I", CSRC, "-o", exe, os.path.join(HERE, "launch_rules_host.cu")])

    def ask(*args):
        out = subprocess.run([exe], input=" ".join(str(a) for a in args) + "\n", capture_output=True, text=True, check=True)
        return tuple(int(x) for x in out.stdout.split())

    return ask


# (two words of 384 x 384 took 43 us a sweep in 768 tiles of 8 rows, 39 in 384 of 16; 100 x 100 is the other way round)
@pytest.mark.parametrize("L,Lc,words,rows", [(384, 384, 2, 16), (192, 192, 8, 16), (96, 96, 32, 16), (96, 96, 24, 8),
                                             (250, 198, 4, 8), (64, 64, 2, 4), (100, 100, 16, 4), (96, 96, 2, 4),
                                             (384, 384, 24, 16), (4, 4, 2, 4)])
def test_streamed_tile_rows(rule, L, Lc, words, rows):
    seg, r = rule("rows", L, Lc, words)
    assert r == rows and 4 <= seg <= 6


def test_streamed_tiles_cover_every_lattice(rule):
    """Rows and segments within the kernels' shared memory, at any size."""
    for L, Lc, words in [(4, 4096, 2), (4096, 4, 2), (4096, 4096, 2), (6, 8, 65534), (1000, 998, 300)]:
        for cut in ("rows", "count"):
            seg, r = rule(cut, L, Lc, words)
            assert r in (4, 8, 16) and seg in (4, 5, 6)


# (the CTAs of a word add their counts to the same 96 addresses: 704 tiles of two words of 256 x 256 took 43 us a sweep
# with its count, 176 take 37)
@pytest.mark.parametrize("L,Lc,words,rows", [(256, 256, 2, 16), (384, 384, 2, 16), (512, 512, 2, 16), (192, 192, 8, 16),
                                             (100, 100, 2, 4), (64, 64, 2, 4), (100, 100, 32, 8)])
def test_streamed_count_rows(rule, L, Lc, words, rows):
    assert rule("count", L, Lc, words)[1] == rows


# sweeps, words, cells, CTAs per SM of the persistent grid, resident CTAs of a CTA per word: a one-sweep launch of 1600
# words of L = 4 took 191 us through the scheduler, 46 with a CTA per word; long launches balance the SMs in chunks
@pytest.mark.parametrize("sweeps,words,cells,per_sm,resident,everything", [
    (1, 1600, 4, 4, 4, 1), (1, 1600, 9, 4, 4, 1), (4, 384, 9, 2, 4, 1), (1, 250, 81, 1, 2, 1), (4, 384, 81, 2, 3, 1),
    (1, 384, 225, 2, 2, 1), (265, 600, 49, 2, 2, 1), (500, 384, 81, 2, 3, 0), (2000, 384, 81, 2, 3, 0), (500, 250, 81, 1, 2, 0)])
def test_short_launches_take_a_cta_per_word(rule, sweeps, words, cells, per_sm, resident, everything):
    every, chunk = rule("schedule", sweeps, words, cells, per_sm, resident)
    assert every == everything
    assert chunk == sweeps if every else 1 <= chunk < sweeps


def test_schedule_chunks_at_any_size(rule):
    for args in [(1, 153, 4, 1, 1), (1 << 20, 1 << 20, 2304, 1, 1), (7, 100000, 4, 4, 4), (1 << 20, 153, 4, 4, 4)]:
        every, chunk = rule("schedule", *args)
        assert 1 <= chunk <= args[0] and (not every or chunk == args[0])


# with 4 warps 1600 words of L = 4 are not all resident and took 9.1 us a sweep, with 3 4.4; 3000 words 12.3, with 1 7.5
@pytest.mark.parametrize("L,words,warps", [(4, 1600, 3), (6, 1600, 3), (8, 1600, 3), (4, 3000, 1), (6, 3000, 1), (8, 3000, 1),
                                           (10, 3000, 3), (12, 1600, 4), (4, 800, 4), (8, 1300, 4), (18, 1600, 8), (18, 384, 14),
                                           (48, 250, 16), (48, 160, 16), (40, 250, 16), (4, 250, 4)])
def test_bitplane_warps(rule, L, words, warps):
    assert rule("bitplane", L, L, words) == (warps,)


# warps of the largest member, CTAs, shared memory of a CTA: 1200 CTAs of half words of L = 12 took 37.9 us a sweep at 12
# warps, a CTA per SM, and 14.9 at 4, four per SM; L = 48 (170 KB) is alone on its SM at any size
@pytest.mark.parametrize("warps,ctas,smem,chosen", [(12, 1200, 56320, 4), (16, 120, 174000, 16), (16, 480, 174000, 16), (16, 152, 57000, 16),
                                                    (16, 160, 60000, 8), (16, 1600, 95000, 8), (4, 800, 56320, 4), (16, 400, 70000, 4)])
def test_batch_warps(rule, warps, ctas, smem, chosen):
    assert rule("batch", warps, ctas, smem) == (chosen,)


# a sweep and a sample of 384 words of L = 48 took 1730 us with 16 warps (1140 before the row form), 1133 with 32
@pytest.mark.parametrize("L,words,correlations,warps", [(48, 384, 1, 32), (36, 1, 1, 32), (96, 2, 1, 32), (34, 1, 1, 16), (18, 384, 1, 8),
                                                        (18, 384, 0, 8), (48, 384, 0, 16), (36, 96, 0, 16), (6, 2, 0, 12)])
def test_canonical_warps(rule, L, words, correlations, warps):
    assert rule("canonical", L, L, words, correlations) == (warps,)
