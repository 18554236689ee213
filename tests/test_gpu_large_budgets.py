"""q = 6 reads whose budgets are too large for token look-ups: their bins' vectors
are checked whole, in candidate lists and among the coarse pass's survivors."""
import numpy as np
import pytest

import oracle
from tests.conftest import Reads
from tests.gpu_helpers import assert_same, build, gpu_filter

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _genome(n, seed):
    rng = np.random.default_rng(seed)
    g = rng.choice(np.frombuffer(b"ACGT", np.uint8), n)
    g[n // 2:n // 2 + 2000] = np.tile(g[:125], 16)
    g[n // 3:n // 3 + 600] = ord("A")
    g[n // 4:n // 4 + 600] = np.resize(np.frombuffer(b"CA", np.uint8), 600)
    return g


def _reads(g, L, n):
    """Random places, the repeat, one repeated base, a two-base repeat, non-bases."""
    rng = np.random.default_rng(L + n)
    at = rng.integers(0, len(g) - L, n)
    at[:4] = len(g) // 2 + 7, len(g) // 3 + 5, len(g) // 4 + 3, len(g) // 3 + 600 - L // 2
    reads = [g[p:p + L].tobytes().decode() for p in at]
    reads[4] = reads[4][:L // 2] + "n" * (L - L // 2)
    reads[5] = "N" + reads[5][1:]
    return reads


@pytest.mark.parametrize("L", [133, 134, 150, 197, 260])
@pytest.mark.parametrize("far", [5, 6, 18])
def test_lists_of_large_budgets(L, far):
    """18 reads of which `far` have budgets past the look-ups (from a third of the
    batch on they are checked whole; reads of 128 tokens never are), from there to
    T <= 0, the others small ones; lists of 0, 1, 31, 32, 33, 100 and more."""
    g = _genome(40_000, L)
    reads = _reads(g, L, 18)
    big = [19, 20, 22, 25, 33, 300]
    e = [big[i % 6] if i < far else i % 8 for i in range(18)]
    order = np.random.default_rng(far).permutation(18)
    e = [e[i] for i in order]
    rng = np.random.default_rng(L * 100 + far)
    counts = [400, 400, 400, 33, 31, 32, 1, 0, 100, 64, 5, 0, 400, 96, 97, 3, 400, 32]
    nb = -(-len(g) // 100)
    cand = np.concatenate([rng.integers(0, nb, c) for c in counts]).astype(np.int32)
    off = np.concatenate([[0], np.cumsum(counts)]).astype(np.uint64)
    cand[:400] = np.arange(400) % nb
    rs = Reads(reads, e)
    ix = build(g, 100, 6, 260, layouts=2)
    want = oracle.filter(oracle.bin_vectors(g, 100, 6, 260), rs, cand_off=off, cand=cand)
    assert len(want[0]) > 100
    assert_same(gpu_filter(ix, rs, off, cand, cap=4000), want)
    bad = cand.copy()
    bad[off[3].astype(int)] = nb
    from paper_1708_04329_gb300 import grim
    with pytest.raises(grim.GrimError) as ei:
        gpu_filter(ix, rs, off, bad, cap=4000)
    assert ei.value.code == grim.GRIM_E_BAD_CANDIDATE
    ix.close()


@pytest.mark.parametrize("factor,L", [(7, 150), (8, 150), (16, 37), (16, 250), (33, 200), (64, 250)])
def test_survivors_of_large_budgets(factor, L):
    """Survivors of reads with D' below, at and past the line, up to where every
    bin passes, and super-bins of fewer members at the end; one path forced."""
    from paper_1708_04329_gb300 import grim

    g = _genome(100 * factor * 41 + 11, factor)
    reads = _reads(g, L, 60)
    e = [(5, 6, L // 10, L // 8, L // 6 + 1, 2, L // 5)[i % 7] for i in range(60)]
    rs = Reads(reads, e)
    ix = build(g, 100, 6, 260, layouts=6, coarse_factor=factor)
    nb = ix.desc.num_bins
    want = oracle.filter(oracle.bin_vectors(g, 100, 6, 260), rs)
    assert len(want[0]) > nb
    assert_same(gpu_filter(ix, rs, cap=60 * nb), want)
    assert grim.grim_last_filter_stats()["survivors"] > 0
    ix.close()
