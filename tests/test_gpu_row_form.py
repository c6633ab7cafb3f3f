"""The canonical SMEM sweep's row form (segments of one to three cells of a row
of cells per word, crbm_row_core.cuh) against the oracle, bit for bit: rows cut
into segments of every length, one segment per row (its own right neighbour), and
the lattices whose hidden words or visible draws are kept in their smaller forms;
with two words (split into bands over a cluster from 40 cells up) and with 80
(a CTA each)."""
import numpy as np
import pytest

import paper_2511_20911_gb300 as crbm
from paper_2511_20911_gb300 import workloads

pytestmark = pytest.mark.gpu
EXACT, PAPER = crbm.CRBM_PRECISION_EXACT, crbm.CRBM_PRECISION_PAPER


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    crbm.load_library()


def check(orc, L, Lc, precision, n, splits, warps, monkeypatch):
    monkeypatch.setenv("CRBM_WARPS", str(warps))
    params = workloads.random_params(np.random.default_rng(L * 97 + Lc), 3)
    cp = (np.arange(n) % 3).astype(np.int32)
    s = crbm.Sampler(L, params, n, chain_param=cp, seed=L + Lc, L_cols=Lc, measure_every=1, precision=precision,
                     layout=crbm.CRBM_LAYOUT_SMEM)
    ids = np.arange(n, dtype=np.uint32)
    spins = orc.init_spins((L, Lc), ids, L + Lc)
    sums, t = None, 0
    for k in splits:
        s.sweep(k)
        sums, _, _ = orc.run((L, Lc), params, cp, spins, L + Lc, t, k, 1, chain_ids=ids, periodic=(True, True), sums=sums,
                             precision=precision)
        t += k
        assert np.array_equal(s.get_spins(), spins), f"spins after {t} sweeps"
    assert np.array_equal(s.observables(), sums)


# one segment per row (4, 6 columns), segments of 2 + 2, 3 + 2, 3 + 3 + 1 cells and of single cells (many warps)
@pytest.mark.parametrize("n", [37, 2530])
@pytest.mark.parametrize("precision", [EXACT, PAPER])
@pytest.mark.parametrize("L,Lc,warps", [(4, 4, 1), (4, 6, 3), (6, 4, 9), (8, 8, 2), (8, 10, 4), (10, 14, 5), (14, 10, 32),
                                        (30, 22, 8)])
def test_segment_lengths(orc, L, Lc, warps, precision, n, monkeypatch):
    check(orc, L, Lc, precision, n, [1, 6], warps, monkeypatch)


# records from global memory (64 x 64, 18 x 96: long rows), 16-bit hidden words (68, 76), visible draws made twice (38 x 52)
@pytest.mark.parametrize("n", [33, 2530])
@pytest.mark.parametrize("L,Lc,precision", [(64, 64, EXACT), (18, 96, EXACT), (68, 68, EXACT), (76, 76, EXACT),
                                            (56, 96, EXACT), (38, 52, PAPER), (18, 96, PAPER)])
def test_large_lattices(orc, L, Lc, precision, n, monkeypatch):
    check(orc, L, Lc, precision, n, [2], 16, monkeypatch)


@pytest.mark.parametrize("ladders,precision", [(1, EXACT), (3, PAPER), (17, EXACT)])
def test_split_ladders_match_whole_words(orc, ladders, precision):
    """Few ladders run split over clusters; the same ladders as members of a context of 96 run whole."""
    L, n = 18, 32 * ladders
    beta = list(0.25 * 32.0 ** (np.arange(32) / 31.0))
    params = dict(J=[1.0] * 32, Jp=[1.5] * 32, h=[1.0] * 32, beta=beta)
    kw = dict(seed=5, measure_every=1, swap_every=2, series_len=6, precision=precision)
    few = crbm.Sampler(L, params, n, chain_param=np.tile(np.arange(32), ladders).astype(np.int32), **kw)
    many = crbm.Sampler(L, params, 32 * 96, chain_param=np.tile(np.arange(32), 96).astype(np.int32), **kw)
    for s in (few, many):
        s.set_targets([-16 * L * L] * 32)
        s.sweep(5)
        s.sweep(4)
    assert np.array_equal(few.get_spins(), many.get_spins()[:n])
    assert np.array_equal(few.observables(), many.observables()[:n])
    assert np.array_equal(few.series(), many.series()[:, :n])
    assert np.array_equal(few.permutation(), many.permutation()[:n])
    assert np.array_equal(few.first_hits(), many.first_hits()[:n])


@pytest.mark.parametrize("L,words,precision,splits", [(4, 161, EXACT, [1, 2, 40]), (6, 310, PAPER, [1, 40]), (4, 700, EXACT, [1, 3, 30]),
                                                      (18, 160, EXACT, [1, 3]), (30, 305, PAPER, [1, 2])])
def test_more_words_than_ctas(orc, L, words, precision, splits, monkeypatch):
    """Short launches give every word a CTA, long ones claim chunks of words from a persistent grid."""
    monkeypatch.delenv("CRBM_WARPS", raising=False)
    n = 32 * words - 5
    params = workloads.random_params(np.random.default_rng(L + words), 3)
    cp = (np.arange(n) // 7 % 3).astype(np.int32)
    s = crbm.Sampler(L, params, n, chain_param=cp, seed=words, measure_every=2, precision=precision)
    ids = np.arange(n, dtype=np.uint32)
    spins, sums, t = orc.init_spins(L, ids, words), None, 0
    for k in splits:
        s.sweep(k)
        sums, _, _ = orc.run(L, params, cp, spins, words, t, k, 2, chain_ids=ids, sums=sums, precision=precision)
        t += k
        assert np.array_equal(s.get_spins(), spins), f"spins after {t} sweeps"
    assert np.array_equal(s.observables(), sums)


# records from global memory and 16-bit hidden words, more words than CTAs: a CTA's second word finds the first's expansion table
@pytest.mark.parametrize("L,precision", [(64, EXACT), (68, EXACT), (38, PAPER), (52, PAPER)])
def test_large_lattices_on_a_persistent_grid(L, precision, monkeypatch):
    """A context of 170 words against the same chains in a context of 2 (split, or a CTA per word)."""
    monkeypatch.delenv("CRBM_WARPS", raising=False)
    params = workloads.random_params(np.random.default_rng(L), 3)
    cp = (np.arange(32 * 170) % 3).astype(np.int32)
    many = crbm.Sampler(L, params, 32 * 170, chain_param=cp, seed=9, measure_every=3, precision=precision)
    few = crbm.Sampler(L, params, 64, chain_param=cp[:64], seed=9, measure_every=3, precision=precision)
    for s in (many, few):
        s.sweep(1)
        s.sweep(60)
    assert np.array_equal(many.get_spins()[:64], few.get_spins())
    assert np.array_equal(many.observables()[:64], few.observables())


@pytest.mark.parametrize("L,n", [(36, 40), (48, 33), (68, 32)])
def test_correlations_of_a_large_lattice(L, n, monkeypatch):
    """One sample, after the last sweep, against the spins read back (CTAs of 32 warps beyond L = 34)."""
    monkeypatch.delenv("CRBM_WARPS", raising=False)
    monkeypatch.setenv("CRBM_AUTOTUNE_CACHE", "/nonexistent/none.txt")
    params = workloads.random_params(np.random.default_rng(L), 3)
    cp = (np.arange(n) % 3).astype(np.int32)
    s = crbm.Sampler(L, params, n, chain_param=cp, seed=L, measure_every=2, sq_every=5)
    assert s.warps == 32
    s.sweep(5)
    v = s.get_spins().astype(np.int64)
    corr, samples = s.correlations()
    assert np.array_equal(samples, np.bincount(cp, minlength=3))
    for dR, dC in [(0, 0), (0, 1), (1, 0), (L // 2, L // 2), (L - 1, 3), (7, L - 2), (L // 2 - 1, 33)]:
        c = (v * np.roll(v, (-dR, -dC), axis=(1, 2))).sum(axis=(1, 2))
        assert np.array_equal(corr[:, dR, dC], np.bincount(cp, c, minlength=3).astype(np.int64)), (dR, dC)


@pytest.mark.parametrize("L,Lc,precision", [(14, 14, EXACT), (14, 14, PAPER), (4, 20, EXACT), (20, 4, EXACT), (12, 14, PAPER)])
def test_words_split_in_two(orc, L, Lc, precision, monkeypatch):
    """40 to 79 cells: bands of half the rows, each the other's neighbour above and below (two rows of cells: of one row)."""
    check(orc, L, Lc, precision, 64, [1, 2, 5], 8, monkeypatch)
