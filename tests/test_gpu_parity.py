"""Parity of the CUDA path (through the C-ABI) with the CPU oracle.

Integer work: every comparison is bit-exact -- tables byte for byte, pass
lists record for record (read, bin, count) in order.
"""
import numpy as np
import pytest

import oracle
from tests.conftest import Reads, load_fixture, random_case
from tests.gpu_helpers import assert_same, build, dev_reads, gpu_filter

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


def _np(s: str) -> np.ndarray:
    return np.frombuffer(s.encode(), dtype=np.uint8).copy()


def _gpu_tables(idx, q):
    tm = idx.token_major()
    bm = idx.bin_major()
    return (None if tm is None else tm.cpu().numpy().view(np.uint32),
            None if bm is None else bm.cpu().numpy().view(np.uint32))


def _check_tables(ref: np.ndarray, B: int, q: int, mrl: int, layouts: int = 7, factor: int = 0):
    idx = build(ref, B, q, mrl, layouts, factor)
    tm, bm = _gpu_tables(idx, q)
    oix = oracle.bin_vectors(ref, B, q, mrl)
    vb = oracle.vector_bytes(q)
    if bm is not None:
        got = bm.view(np.uint8).reshape(oix.num_bins, -1)
        assert np.array_equal(got[:, :vb], oix.vecs)
        assert not got[:, vb:].any()
    if tm is not None:
        assert np.array_equal(tm, oracle.token_major(oix))
    ctm = idx.coarse_token_major()
    if ctm is not None:
        # super-bins of f bins: the oracle's vectors with core f*B, same extension
        f = idx.desc.coarse_factor
        coarse = oracle.bin_vectors(ref, f * B, q, mrl)
        assert np.array_equal(ctm.cpu().numpy().view(np.uint32), oracle.token_major(coarse))
        assert idx.desc.num_coarse == coarse.num_bins
    d = idx.desc
    assert d.num_bins == oix.num_bins and d.num_bins_pad % 1024 == 0
    return idx, oix


# ---------------------------------------------------------------------------
# tables (a1-a3)
# ---------------------------------------------------------------------------

def test_fig2_bits_on_gpu():
    fx = load_fixture("fig2_q5.txt")
    idx = build(_np(fx["ref"]), fx["B"], fx["q"], fx["max_read_len"])
    tm, bm = _gpu_tables(idx, 5)
    bits = np.unpackbits(bm.view(np.uint8)[0], bitorder="little")
    assert sorted(np.flatnonzero(bits).tolist()) == sorted(fx["set"])
    for t in fx["set"]:
        assert tm[t, 0] & 1
    for t in fx["clear"]:
        assert not tm[t, 0] & 1


@pytest.mark.parametrize("q", [2, 3, 4, 5, 6])
def test_tables_match_oracle(q):
    rng = np.random.default_rng(100 + q)
    n = int(rng.integers(20_000, 60_000))
    B = int(rng.integers(7, 40))
    ref, _, _ = random_case(rng, q, n, B, 50, 0)
    _check_tables(_np(ref), B, q, int(rng.integers(q, 80)))


def test_tables_ragged_and_tiny():
    # one base shorter than q, a single bin, a window clipped at N
    for ref, B, q, mrl in [("ACG", 5, 4, 4), ("ACGTA", 5, 4, 10), ("ACGTACGTNNacgtTT", 3, 3, 5)]:
        _check_tables(_np(ref), B, q, mrl)


def test_build_host_equals_build():
    from paper_1708_04329_gb300 import grim

    g = np.frombuffer(b"ACGT", np.uint8)[np.random.default_rng(3).integers(0, 4, 70_001)]
    a = build(g, 50, 5, 100)
    b = grim.grim_build_host(g, 50, 5, 100)
    assert np.array_equal(a.token_major().cpu().numpy(), b.token_major().cpu().numpy())
    assert np.array_equal(a.bin_major().cpu().numpy(), b.bin_major().cpu().numpy())


# ---------------------------------------------------------------------------
# filter (a4-a8)
# ---------------------------------------------------------------------------

def test_handworked_fixture_gpu():
    fx = load_fixture("handworked_q3.txt")
    rs = Reads([r for r, _ in fx["read"]], [x for _, x in fx["read"]])
    idx = build(_np(fx["ref"]), fx["B"], fx["q"], fx["max_read_len"])
    r, b, c = gpu_filter(idx, rs)
    assert list(zip(r.tolist(), b.tolist(), c.tolist())) == fx["pass"]


@pytest.mark.parametrize("layouts", [1, 6, 7])
@pytest.mark.parametrize("seed", range(8))
def test_random_all_bins(seed, layouts):
    """Several 1024-bin tiles plus a ragged one, mixed read lengths, non-bases,
    per-read e including T <= 0; one exact pass over the token-major table
    (layouts 1), coarse-then-exact (6), or whichever the batch suits (7)."""
    rng = np.random.default_rng(500 + seed)
    q = int(rng.choice([2, 3, 4, 5, 6]))
    B = int(rng.integers(5, 40))
    mrl = int(rng.integers(max(q, 20), 120))
    n = int(rng.integers(30_000, 90_000))
    ref, reads, e = random_case(rng, q, n, B, mrl, 300)
    if seed % 2:  # half the cases with some T <= 0 reads
        e = [int(x) if rng.random() < 0.9 else 40 for x in e]
    rs = Reads(reads, e)
    idx, oix = _check_tables(_np(ref), B, q, mrl, layouts)
    assert_same(gpu_filter(idx, rs), oracle.filter(oix, rs))


@pytest.mark.parametrize("seed", range(6))
def test_random_candidates(seed):
    """Unsorted lists with duplicates and empty lists keep the given order."""
    rng = np.random.default_rng(700 + seed)
    q = int(rng.choice([2, 3, 4, 5, 6]))
    B = int(rng.integers(5, 40))
    mrl = int(rng.integers(max(q, 20), 120))
    n = int(rng.integers(20_000, 60_000))
    ref, reads, e = random_case(rng, q, n, B, mrl, 300)
    rs = Reads(reads, e)
    idx, oix = _check_tables(_np(ref), B, q, mrl)
    nb = oix.num_bins
    counts = rng.integers(0, 40, len(reads))
    counts[rng.random(len(reads)) < 0.1] = 0
    off = np.zeros(len(reads) + 1, np.uint64)
    off[1:] = np.cumsum(counts)
    cand = rng.integers(0, nb, int(off[-1])).astype(np.int32)
    assert_same(gpu_filter(idx, rs, off, cand), oracle.filter(oix, rs, cand_off=off, cand=cand))


def test_tiny_plain_full(tiny_plain, tiny_plain_index, tiny_plain_oracle):
    """The 1 Mbp / 5,000-bin / 2,000-read workload: the whole pass list."""
    w = tiny_plain
    idx = build(w["genome"], w["B"], w["q"], w["max_read_len"])
    assert_same(gpu_filter(idx, w["reads"]), tiny_plain_oracle)
    from paper_1708_04329_gb300 import synth

    off, cand = synth.candidates((w["reads"].true_pos // w["B"]).astype(np.int32),
                                 tiny_plain_index.num_bins, seed=4)
    assert_same(gpu_filter(idx, w["reads"], off, cand),
                oracle.filter(tiny_plain_index, w["reads"], cand_off=off, cand=cand))


def test_many_ranges_per_tile():
    """Few tiles, many reads: each tile is split into read ranges."""
    from paper_1708_04329_gb300 import synth

    g = synth.genome(250_000, seed=9)
    rs = synth.reads(g, 6000, seed=10, e=5, max_edits=5)
    idx = build(g, 200, 5, 100)
    oix = oracle.bin_vectors(g, 200, 5, 100)
    assert_same(gpu_filter(idx, rs), oracle.filter(oix, rs))


def test_threshold_nonpositive_passes_everything():
    from paper_1708_04329_gb300 import synth

    g = synth.genome(40_000, seed=5)
    rs = synth.reads(g, 7, seed=6, e=20, max_edits=5)
    idx = build(g, 100, 5, 100)
    oix = oracle.bin_vectors(g, 100, 5, 100)
    got = gpu_filter(idx, rs)
    assert len(got[0]) == 7 * oix.num_bins
    assert_same(got, oracle.filter(oix, rs))


def test_reads_of_every_length_in_one_call():
    rng = np.random.default_rng(11)
    ref, _, _ = random_case(rng, 5, 50_000, 64, 0, 0, dirty=False)
    g = _np(ref)
    reads = []
    for L in range(5, 256):
        s = int(rng.integers(0, len(ref) - L))
        reads.append(ref[s:s + L])
    rs = Reads(reads, [int(x) for x in rng.integers(0, 6, len(reads))])
    idx = build(g, 64, 5, 255)
    oix = oracle.bin_vectors(g, 64, 5, 255)
    want = oracle.filter(oix, rs)
    assert_same(gpu_filter(idx, rs), want)
    # and with every read switch and both all-bins paths forced: under the
    # warp switch the groups of a warp end 1 to 16 blocks apart, so groups
    # whose read ended read on through their token rows' padding
    from paper_1708_04329_gb300 import grim

    for path in (grim.GRIM_PATH_TWO_LEVEL, grim.GRIM_PATH_EXACT):
        for switch in (grim.GRIM_SWITCH_GROUP, grim.GRIM_SWITCH_WARP):
            grim.grim_index_set_shape(idx, read_switch=switch, all_bins_path=path)
            assert_same(gpu_filter(idx, rs), want)
    # reversed length order: long and short reads share every warp
    back = Reads(reads[::-1], list(rs.e[::-1]))
    grim.grim_index_set_shape(idx, read_switch=grim.GRIM_SWITCH_WARP)
    assert_same(gpu_filter(idx, back), oracle.filter(oix, back))
    idx.close()


def test_zero_reads():
    from paper_1708_04329_gb300 import grim

    idx = build(_np("ACGTACGTAC" * 10), 10, 3, 10)
    z = torch.zeros(0, dtype=torch.int64, device="cuda")
    r, b, c = grim.grim_filter(idx, torch.zeros(0, dtype=torch.uint8, device="cuda"), z,
                               z.to(torch.int32), z.to(torch.int16))
    assert r.numel() == 0


@pytest.mark.parametrize("reads,code", [(["ACGTAC", "AC"], -4), (["ACGTACGTACGT"], -5),
                                        (["AC", "ACGTACGTACGT"], -4)])
def test_read_length_errors(reads, code):
    from paper_1708_04329_gb300 import grim

    idx = build(_np("ACGTACGTAC" * 10), 10, 3, 10)
    with pytest.raises(grim.GrimError) as ei:
        gpu_filter(idx, Reads(reads, [0] * len(reads)))
    assert ei.value.code == code


def test_candidate_errors():
    from paper_1708_04329_gb300 import grim

    idx = build(_np("ACGTACGTAC" * 10), 10, 3, 10)
    rs = Reads(["ACGTAC", "CGTACG"], [0, 0])
    with pytest.raises(grim.GrimError) as ei:
        gpu_filter(idx, rs, np.array([0, 1, 2], np.uint64), np.array([3, 10], np.int32))
    assert ei.value.code == grim.GRIM_E_BAD_CANDIDATE
    with pytest.raises(grim.GrimError) as ei:  # decreasing offsets
        gpu_filter(idx, rs, np.array([0, 2, 1], np.uint64), np.array([3, 4], np.int32))
    assert ei.value.code == grim.GRIM_E_ARG
    # an index with only the token-major table cannot serve candidate lists
    tmo = build(_np("ACGTACGTAC" * 10), 10, 3, 10, layouts=1)
    with pytest.raises(grim.GrimError) as ei:
        gpu_filter(tmo, rs, np.array([0, 1, 2], np.uint64), np.array([3, 4], np.int32))
    assert ei.value.code == grim.GRIM_E_NO_LAYOUT


def test_overflow_reports_total_and_count_only():
    from paper_1708_04329_gb300 import grim, synth
    from tests.gpu_helpers import dev_reads

    g = synth.genome(40_000, seed=5)
    rs = synth.reads(g, 50, seed=6, e=5, max_edits=5)
    idx = build(g, 100, 5, 100)
    want = oracle.filter(oracle.bin_vectors(g, 100, 5, 100), rs)
    n = len(want[0])
    assert n > 3
    for cap in (0, 3):
        out = tuple(torch.empty(cap, dtype=dt, device="cuda")
                    for dt in (torch.int32, torch.int32, torch.uint8))
        with pytest.raises(grim.GrimError) as ei:
            grim.grim_filter(idx, **dev_reads(rs), out=out)
        assert ei.value.code == grim.GRIM_E_OVERFLOW and ei.value.n_out == n
    # the binding's retry returns the full list
    assert_same(gpu_filter(idx, rs, cap=1), want)
    # coarse-then-exact without a token-major table: an overflow of the
    # survivors reports an upper bound, and the retry with it succeeds
    cto = build(g, 100, 5, 100, layouts=6)
    out = tuple(torch.empty(3, dtype=dt, device="cuda") for dt in (torch.int32, torch.int32, torch.uint8))
    with pytest.raises(grim.GrimError) as ei:
        grim.grim_filter(cto, **dev_reads(rs), out=out)
    assert ei.value.code == grim.GRIM_E_OVERFLOW and ei.value.n_out >= n
    assert_same(gpu_filter(cto, rs, cap=3), want)


def test_workspace_reuse_is_clean():
    from paper_1708_04329_gb300 import grim, synth

    g = synth.genome(80_000, seed=7)
    a = synth.reads(g, 500, seed=8, e=5, max_edits=5)
    b = synth.reads(g, 300, seed=9, e=3, max_edits=3)
    idx = build(g, 200, 5, 100)
    oix = oracle.bin_vectors(g, 200, 5, 100)
    ws = grim.Workspace()
    for rs in (a, b, a):
        assert_same(gpu_filter(idx, rs, workspace=ws), oracle.filter(oix, rs))


def test_filter_host_equals_oracle():
    from paper_1708_04329_gb300 import grim, synth

    g = synth.genome(80_000, seed=12)
    rs = synth.reads(g, 400, seed=13, e=5, max_edits=5)
    idx = build(g, 200, 5, 100)
    oix = oracle.bin_vectors(g, 200, 5, 100)
    got = grim.grim_filter_host(idx, rs.seq, rs.offsets, rs.lens, rs.e)
    assert_same(got, oracle.filter(oix, rs))
    off, cand = synth.candidates((rs.true_pos // 200).astype(np.int32), oix.num_bins, seed=3)
    got = grim.grim_filter_host(idx, rs.seq, rs.offsets, rs.lens, rs.e, cand=cand, cand_off=off)
    assert_same(got, oracle.filter(oix, rs, cand_off=off, cand=cand))


@pytest.mark.parametrize("layouts", [1, 6, 7])
def test_q6_all_bins(layouts):
    """q = 6 (4096-row table, 256-bin tiles): several tiles plus a ragged one."""
    from paper_1708_04329_gb300 import synth

    g = synth.human_genome(400_000, seed=8)
    rs = synth.reads(g, 700, seed=9, lengths=(150,), e=7, max_edits=7)
    idx, oix = _check_tables(g, 100, 6, 150, layouts)
    if layouts & 4:  # default factor: the largest power of two keeping a window near 40% full
        assert idx.desc.coarse_factor == 16
    assert_same(gpu_filter(idx, rs), oracle.filter(oix, rs))


@pytest.mark.parametrize("lengths", [(150,), (60, 150, 250)])
def test_q6_read_switch_modes(lengths):
    """q = 6, every read switch: with sixteen 2-lane groups per warp the warp
    switch takes new reads once 14 groups wait, so the others keep reads that
    started earlier (groups out of phase, token blocks past the slot read
    from L2).  2,400 reads span several read ranges of a 1 MiB read tile;
    uniform and mixed lengths; both all-bins paths; equal to the oracle."""
    from paper_1708_04329_gb300 import grim, synth

    g = synth.human_genome(600_000, seed=12)
    rs = synth.reads(g, 2400, seed=13, lengths=lengths, probs=(1.0,) if len(lengths) == 1 else (0.3, 0.4, 0.3),
                     e_frac=(5, 100), max_edits=None)
    idx = build(g, 100, 6, 250)
    want = oracle.filter(oracle.bin_vectors(g, 100, 6, 250), rs)
    for path in (grim.GRIM_PATH_TWO_LEVEL, grim.GRIM_PATH_EXACT):
        for switch in (grim.GRIM_SWITCH_GROUP, grim.GRIM_SWITCH_WARP, 0):
            grim.grim_index_set_shape(idx, read_range_kb=1024, read_switch=switch, all_bins_path=path)
            assert_same(gpu_filter(idx, rs), want)
    idx.close()


def test_default_coarse_factor_q5():
    from paper_1708_04329_gb300 import synth

    g = synth.genome(50_000, seed=2)
    assert build(g, 200, 5, 100).desc.coarse_factor == 2


@pytest.mark.parametrize("q,factor", [(4, 3), (5, 4), (5, 7), (6, 8), (6, 16)])
def test_coarse_factors(q, factor):
    """Coarse-then-exact with super-bins of 3..16 bins (ragged last super-bin)."""
    rng = np.random.default_rng(900 + factor)
    B = int(rng.integers(20, 60))
    mrl = 120
    ref, reads, e = random_case(rng, q, 90_001, B, mrl, 300)
    rs = Reads(reads, e)
    idx, oix = _check_tables(_np(ref), B, q, mrl, layouts=6, factor=factor)
    assert idx.desc.coarse_factor == factor
    assert_same(gpu_filter(idx, rs), oracle.filter(oix, rs))


def _low_complexity_case(rng, n: int, n_reads: int, mrl: int):
    """A genome with homopolymer and short tandem-repeat blocks, and reads
    drawn from them (or made of such repeats): tokens of high multiplicity,
    up to L-q+1 copies of one token."""
    alpha = np.frombuffer(b"ACGT", dtype=np.uint8)
    g = alpha[rng.integers(0, 4, n)].copy()
    blocks = []
    for period in (1, 1, 2, 3, 4, 6, 7, 8, 12):
        unit = alpha[rng.integers(0, 4, period)]
        size = int(rng.integers(150, 400))
        s = int(rng.integers(0, n - size))
        g[s:s + size] = np.resize(unit, size)
        blocks.append((s, size))
    ref = g.tobytes().decode()
    reads, es = [], []
    for _ in range(n_reads):
        L = int(rng.integers(max(20, mrl // 2), mrl + 1))
        kind = rng.random()
        if kind < 0.5:  # from (or across the edge of) a low-complexity block
            s0, size = blocks[int(rng.integers(0, len(blocks)))]
            s = int(np.clip(s0 + rng.integers(-L // 2, size), 0, n - L))
            rd = bytearray(ref[s:s + L].encode())
            for _k in range(int(rng.integers(0, 3))):
                rd[int(rng.integers(0, L))] = b"ACGT"[int(rng.integers(0, 4))]
        elif kind < 0.8:  # a pure tandem repeat, period 1..8
            unit = alpha[rng.integers(0, 4, int(rng.integers(1, 9)))]
            rd = bytearray(np.resize(unit, L).tobytes())
        else:
            rd = bytearray(alpha[rng.integers(0, 4, L)].tobytes())
        reads.append(rd.decode())
        es.append(int(rng.integers(0, 6)))
    return ref, reads, es, blocks


@pytest.mark.parametrize("q", [5, 6])
def test_repeated_tokens(q):
    """Reads whose tokens repeat many times (homopolymers, short tandem
    repeats): the multiplicity planes above the first two -- in shared
    memory for 128-byte vectors, the list of heavy tokens for 512-byte ones
    -- in candidate mode and in the coarse-then-exact all-bins mode."""
    rng = np.random.default_rng(1100 + q)
    B, mrl = 40, 150
    ref, reads, e, blocks = _low_complexity_case(rng, 60_000, 400, mrl)
    rs = Reads(reads, e)
    idx, oix = _check_tables(_np(ref), B, q, mrl, layouts=7)
    nb = oix.num_bins
    block_bins = np.concatenate([np.arange(s // B, min(nb, (s + size) // B + 1))
                                 for s, size in blocks]).astype(np.int32)
    lists = []
    for _ in reads:
        picks = [rng.integers(0, nb, int(rng.integers(0, 30))),
                 rng.choice(block_bins, int(rng.integers(0, 30)))]
        lists.append(np.concatenate(picks).astype(np.int32))
    off = np.zeros(len(reads) + 1, np.uint64)
    off[1:] = np.cumsum([len(x) for x in lists])
    cand = np.concatenate(lists).astype(np.int32)
    want = oracle.filter(oix, rs, cand_off=off, cand=cand)
    assert len(want[0]) > 100  # the repeats do pass somewhere
    assert_same(gpu_filter(idx, rs, off, cand), want)
    assert_same(gpu_filter(idx, rs), oracle.filter(oix, rs))


@pytest.mark.parametrize("layouts", [1, 6, 7])
def test_degenerate_genome_and_reads(layouts):
    """A genome of non-bases (no bin holds any q-gram: only reads with T <= 0
    pass, with count 0) and a read of non-bases against a clean genome, in
    the all-bins paths and in candidate mode."""
    q, B, mrl = 4, 10, 20
    reads = ["ACGTACGTAC", "NNNNNNNNNN", "ACGTNACGTA", "acgtacgtac", "NNNNNNNNNNNNNNNNNNNN"]
    for ref, e in (("N" * 2_095, [0, 2, 2, 3, 5]), ("ACGTTGCAAC" * 300, [1, 2, 0, 1, 5]),
                   ("ACGTTGCAAC" * 300, [0, 1, 1, 0, 4])):
        rs = Reads(reads, e)
        idx, oix = _check_tables(_np(ref), B, q, mrl, layouts)
        assert_same(gpu_filter(idx, rs), oracle.filter(oix, rs))
        if layouts & 2:
            nb = oix.num_bins
            off = np.array([0, 3, 3, 7, 9, 12], np.uint64)
            cand = np.array([0, 1, nb - 1, 5, 4, 3, 2, 0, nb - 1, 7, 8, 9], np.int32)
            assert_same(gpu_filter(idx, rs, off, cand), oracle.filter(oix, rs, cand_off=off, cand=cand))
        idx.close()


def test_filter_stats_are_per_thread():
    """grim_last_filter_stats reports the calling thread's own last call:
    two threads filtering different batches at the same time (each on its
    own stream and workspace) each read back the counters of their own call,
    identical to the same call made alone."""
    import threading

    from paper_1708_04329_gb300 import grim, synth

    torch.cuda.set_device(0)
    g = synth.human_genome(1_500_000, seed=91)
    idx = build(g, 200, 5, 100)
    batches = [synth.reads(g, 3000, seed=92, e=5, max_edits=5),
               synth.reads(g, 1200, seed=93, e=3, max_edits=3)]
    alone = []
    for rs in batches:
        grim.grim_filter(idx, **dev_reads(rs))
        alone.append(grim.grim_last_filter_stats())
    assert alone[0] != alone[1]
    got = [None, None]
    errors = []

    def work(i):
        try:
            st = torch.cuda.Stream()
            ws = grim.Workspace()
            kw = dev_reads(batches[i])
            for _ in range(5):
                with torch.cuda.stream(st):
                    grim.grim_filter(idx, **kw, workspace=ws, stream=st)
                s = grim.grim_last_filter_stats()
                if s != alone[i]:
                    errors.append((i, s))
            got[i] = s
        except Exception as e:  # surfaced below
            errors.append((i, repr(e)))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    assert got == alone
    idx.close()


@pytest.mark.parametrize("path", ["exact", "two_level"])
def test_one_word_tail(path):
    """With the warp-synchronous read switch, a warp whose lanes each hold at
    most one word (32 bins) with a live bin after four blocks applies its
    remaining blocks to that word alone.  On repeat-rich 100 bp reads (6
    blocks each) most warps get there; the counters show it (fewer bit tests
    than tokens x tile bins) and the pass list stays exactly the oracle's, and
    equal to the group switch, which never takes the tail.  15,000 bins end
    in a ragged tile (15 x 1024 = 15,360)."""
    from paper_1708_04329_gb300 import grim, synth

    g = synth.human_genome(3_000_000, seed=95)
    rs = synth.reads(g, 4000, seed=96, lengths=(100,), e=5, max_edits=5)
    idx = build(g, 200, 5, 100)
    assert idx.desc.num_bins == 15000
    p = grim.GRIM_PATH_EXACT if path == "exact" else grim.GRIM_PATH_TWO_LEVEL
    want = oracle.filter(oracle.bin_vectors(g, 200, 5, 100), rs)
    got = {}
    for switch in (grim.GRIM_SWITCH_WARP, grim.GRIM_SWITCH_GROUP):
        grim.grim_index_set_shape(idx, read_switch=switch, all_bins_path=p)
        got[switch] = gpu_filter(idx, rs)
        st = grim.grim_last_filter_stats()
        full = st["tokens_executed"] * 1024
        if switch == grim.GRIM_SWITCH_WARP:
            assert st["bit_tests_executed"] < full  # the tail ran
        else:
            assert st["bit_tests_executed"] == full
    assert_same(got[grim.GRIM_SWITCH_WARP], want)
    assert_same(got[grim.GRIM_SWITCH_GROUP], want)
    idx.close()


def test_automatic_read_switch_and_path():
    """The choices a call makes on its own, reported by grim_last_filter_stats:
    the warp switch only when every read spans as many 16-token blocks and
    has the same miss budget D' (with budgets that differ, reads leave a tile
    blocks apart); coarse-then-exact unless a read has too little slack.  The
    pass list equals the oracle's in every case."""
    from paper_1708_04329_gb300 import grim, synth

    g = synth.human_genome(1_000_000, seed=97)
    idx = build(g, 200, 5, 150)
    oix = oracle.bin_vectors(g, 200, 5, 150)
    W, G = grim.GRIM_SWITCH_WARP, grim.GRIM_SWITCH_GROUP
    two, exact = grim.GRIM_PATH_TWO_LEVEL, grim.GRIM_PATH_EXACT
    cases = [
        (synth.reads(g, 1500, seed=98, lengths=(100,), e=5, max_edits=5), W, two),
        (synth.reads(g, 1500, seed=99, lengths=(100,), e_frac=(5, 100), max_edits=None), G, two),
        (synth.reads(g, 1500, seed=100, lengths=(100, 150), probs=(0.5, 0.5), e=5, max_edits=5), G, two),
        # 96 tokens, D' = 75: slack 21 < 24, so the exact pass
        (synth.reads(g, 600, seed=101, lengths=(100,), e=15, max_edits=3), W, exact),
    ]
    for rs, switch, path in cases:
        assert_same(gpu_filter(idx, rs), oracle.filter(oix, rs))
        st = grim.grim_last_filter_stats()
        assert (st["read_switch"], st["all_bins_path"]) == (switch, path)
    # candidate mode reports neither
    off, cand = synth.candidates((cases[0][0].true_pos // 200).astype(np.int32), oix.num_bins, seed=3)
    gpu_filter(idx, cases[0][0], off, cand)
    st = grim.grim_last_filter_stats()
    assert (st["read_switch"], st["all_bins_path"]) == (0, 0)
    idx.close()


def test_survivor_overflow_takes_the_exact_pass():
    """Coarse survivors beyond their room (the larger of the output capacity
    and 320 a read) with the token-major table present: the call drops the
    coarse result and takes the exact pass, reports that path, and still
    equals the oracle.  The genome repeats one random 127-base period: a
    super-bin window (2 x 24 + 79 = 127 bases) holds nearly every q-gram of
    the period, so ~998 super-bins pass per read, while a bin window (103
    bases) holds a read's q-grams only near its copies (~551 bins a read)."""
    from paper_1708_04329_gb300 import grim

    rng = np.random.default_rng(41)
    period = "".join("ACGT"[i] for i in rng.integers(0, 4, 127))
    ref = (period * (48_000 // 127 + 1))[:48_000]
    reads = []
    for _ in range(20):
        s = int(rng.integers(0, len(ref) - 80))
        reads.append(ref[s:s + 80])
    rs = Reads(reads, [1] * len(reads))
    g = _np(ref)
    want = oracle.filter(oracle.bin_vectors(g, 24, 5, 80), rs)
    n_surv = len(oracle.filter(oracle.bin_vectors(g, 48, 5, 80), rs)[0])
    assert n_surv > max(len(want[0]), 320 * rs.n)  # the survivors do not fit
    idx = build(g, 24, 5, 80, coarse_factor=2)
    grim.grim_index_set_shape(idx, all_bins_path=grim.GRIM_PATH_TWO_LEVEL)
    assert_same(gpu_filter(idx, rs, cap=len(want[0])), want)
    st = grim.grim_last_filter_stats()
    assert st["survivors"] == n_surv
    assert st["all_bins_path"] == grim.GRIM_PATH_EXACT
    # with room for every survivor the same call stays on the coarse path
    assert_same(gpu_filter(idx, rs, cap=n_surv), want)
    st = grim.grim_last_filter_stats()
    assert st["survivors"] == n_surv and st["all_bins_path"] == grim.GRIM_PATH_TWO_LEVEL
    idx.close()


@pytest.mark.parametrize("q,factor,n", [(4, 3, 1), (5, 2, 15), (5, 2, 16), (5, 2, 17), (5, 64, 1),
                                        (6, 16, 2), (6, 5, 33)])
def test_survivor_check_batches(q, factor, n):
    """Survivors are checked in warp batches of 32 (survivor, member) items:
    counts below, at and past a batch, factors that cut a survivor across two
    batches, and a last super-bin with fewer members."""
    from paper_1708_04329_gb300 import synth

    g = synth.genome(20 * 64 * 37 + 11, seed=q * 7 + n)
    rs = synth.reads(g, n, seed=n, lengths=(60, 100), probs=(0.5, 0.5), e=3, max_edits=3)
    ix = build(g, 37, q, 100, layouts=6, coarse_factor=factor)
    assert_same(gpu_filter(ix, rs, cap=200_000), oracle.filter(oracle.bin_vectors(g, 37, q, 100), rs))
    ix.close()


@pytest.mark.parametrize("n", [1, 15, 16, 17, 2047, 2048, 2049, 8191, 8192, 8193])
def test_pass_list_order_by_length(n):
    """Pass lists placed by counting smaller keys and by radix sort: one
    record, a block's edge, a shared-memory chunk's edge and the line between
    the two, with unsorted duplicate candidates that all pass (T <= 0)."""
    rng = np.random.default_rng(n)
    g = rng.choice(np.frombuffer(b"ACGT", np.uint8), 60_000)
    nr = max(1, n // 50)
    at = rng.integers(0, len(g) - 40, nr)
    rs = Reads([g[p:p + 40].tobytes().decode() for p in at], [20] * nr)
    cand = rng.integers(0, 1200, n).astype(np.int32)
    off = np.sort(rng.integers(0, n + 1, nr + 1)).astype(np.uint64)
    off[0], off[-1] = 0, n
    ix = build(g, 50, 5, 40, layouts=2)
    got = gpu_filter(ix, rs, off, cand, cap=n)
    assert len(got[0]) == n
    assert_same(got, oracle.filter(oracle.bin_vectors(g, 50, 5, 40), rs, cand_off=off, cand=cand))
    ix.close()


@pytest.mark.parametrize("L", [6, 36, 37, 38, 69, 70, 101, 150, 250, 260])
def test_q6_list_lookups(L):
    """q = 6 lists are ruled out from the first groups of 32 tokens: reads of
    one token, at and past a group's edge and of 255 tokens, budgets from 0
    to T <= 0, reads with non-bases and of one repeated base, lists of 0, 1,
    31, 32, 33 and 100 candidates, duplicates and all bins of a repeat."""
    rng = np.random.default_rng(L)
    g = rng.choice(np.frombuffer(b"ACGT", np.uint8), 40_000)
    g[20_000:22_000] = np.tile(g[:125], 16)
    g[30_000:30_400] = ord("A")
    at = [20_010, 5, 30_050, 1234, 20_300, 39_000 - L, 777, 15_000]
    reads = [g[p:p + L].tobytes().decode() for p in at] * 2
    reads[1] = "N" + reads[1][1:]
    reads[3] = reads[3][:L // 2] + "n" * (L - L // 2)
    e = [0, 1, 2, L // 20, 5, 7, L // 6, 300] + [7] * 8
    counts = [0, 1, 31, 32, 33, 100, 400, 64, 400, 1, 0, 5, 32, 96, 97, 400]
    nb = -(-len(g) // 100)
    cand = np.concatenate([rng.integers(0, nb, c) for c in counts]).astype(np.int32)
    off = np.concatenate([[0], np.cumsum(counts)]).astype(np.uint64)
    cand[off[6].astype(int):off[7].astype(int)] = np.arange(400) % nb
    rs = Reads(reads, e)
    ix = build(g, 100, 6, 260, layouts=2)
    want = oracle.filter(oracle.bin_vectors(g, 100, 6, 260), rs, cand_off=off, cand=cand)
    assert len(want[0]) > 64
    assert_same(gpu_filter(ix, rs, off, cand, cap=2000), want)
    ix.close()


@pytest.mark.parametrize("q,B,mrl,factor,n,layouts,shift", [
    (5, 200, 100, 2, 512 * 200, 7, 0),          # one whole tile, windows of two cores
    (5, 200, 100, 2, 512 * 200 + 1, 7, 1),      # one base into the next; unaligned reference
    (5, 100, 105, 4, 3 * 512 * 100 - 7, 7, 0),  # ext - q + 1 = B: no partial core
    (5, 100, 250, 8, 60_000, 7, 0),             # windows of four cores
    (5, 90, 250, 16, 100_003, 7, 3),
    (5, 61, 250, 2, 40_000, 7, 0),              # more cores than the one-pass build takes
    (5, 173, 101, 3, 120_000, 7, 0),            # a factor whose super-bins do not fill row words
    (5, 200, 100, 2, 300_000, 1, 0),            # single tables
    (5, 200, 100, 2, 300_000, 4, 0),
    (5, 200, 5, 2, 4, 7, 0),                    # shorter than q
    (5, 900, 100, 2, 500_000, 7, 0),            # a tile past shared memory
    (6, 100, 150, 16, 512 * 100 + 37, 7, 0),
    (6, 128, 250, 4, 90_001, 5, 2)])
def test_one_pass_build_shapes(q, B, mrl, factor, n, layouts, shift):
    """Tables of the one-pass build at its tile and window edges, against the
    oracle, with lower case and runs of non-bases; shapes it leaves to the
    other kernels beside them."""
    from paper_1708_04329_gb300 import grim

    rng = np.random.default_rng(n + B)
    g = rng.choice(np.frombuffer(b"ACGTacgt", np.uint8), n)
    for p in rng.integers(0, n, 5):
        g[p:p + int(rng.integers(1, 12))] = ord("N")
    if n > 60_000:
        g[n // 2:n // 2 + 700] = ord("-")
    dev = torch.zeros(n + shift, dtype=torch.uint8, device="cuda")
    dev[shift:] = torch.from_numpy(g).cuda()
    idx = grim.grim_build_ex(dev[shift:], B, q, mrl, layouts, factor)
    oix = oracle.bin_vectors(g, B, q, mrl)
    tm, bm = _gpu_tables(idx, q)
    if bm is not None:
        assert np.array_equal(bm.view(np.uint8).reshape(oix.num_bins, -1), oix.vecs)
    if tm is not None:
        assert np.array_equal(tm, oracle.token_major(oix))
    if layouts & 4:
        coarse = oracle.token_major(oracle.bin_vectors(g, factor * B, q, mrl))
        assert np.array_equal(idx.coarse_token_major().cpu().numpy().view(np.uint32), coarse)
    idx.close()


@pytest.mark.parametrize("B,mrl,factor,n,layouts,shift", [
    (100, 150, 16, 1024 * 16 * 100 + 1, 7, 0),  # one coarse row pad and a base; full tiles
    (100, 150, 8, 512 * 8 * 100 - 3, 7, 1),     # two coarse words a tile
    (90, 250, 8, 200_003, 4, 0),                # super-bins alone, the vectors in scratch
    (128, 150, 16, 70_000, 1, 3),               # rows alone
    (61, 250, 16, 333_333, 6, 0),               # more cores than the one-pass build takes
    (400, 100, 2, 450_000, 7, 0),               # a factor whose vectors have no room
    (900, 6, 8, 512 * 900 + 5, 7, 0)])          # codes larger than the row pieces
def test_one_pass_build_q6_rows(B, mrl, factor, n, layouts, shift):
    """Token rows and super-bins of q = 6 from the one-pass build, against the
    oracle."""
    test_one_pass_build_shapes(6, B, mrl, factor, n, layouts, shift)


@pytest.mark.parametrize("q,B,mrl,layouts", [(5, 50, 250, 7), (5, 50, 100, 1), (6, 100, 150, 6)])
def test_few_reads_on_a_large_table(q, B, mrl, layouts):
    """Batches of a few reads load table rows instead of staging tiles: counts
    up to the rule's line (4 * 4^q rows' worth of tokens) and past it, a last
    tile group cut by the row end, reads of one token, with non-bases and of
    every budget, through the plain call and a plan that holds more reads."""
    from paper_1708_04329_gb300 import grim, synth

    n = 70_000_003
    g = synth.human_genome(n, seed=q)
    ts = -(-(mrl - q + 1) // 16) * 16
    line = 4 * 4 ** q // ts
    rs = synth.reads(g, line + 1, seed=9, lengths=(q, 80, mrl), probs=(0.05, 0.45, 0.5),
                     e_frac=(5, 100), max_edits=None)
    rs.seq[int(rs.offsets[2]) + 3] = ord("N")
    rs.e[rs.lens == q] = 0
    ix = build(g, B, q, mrl, layouts)
    grim.grim_index_set_shape(ix, all_bins_path=0 if layouts != 7 else grim.GRIM_PATH_TWO_LEVEL)
    oix = oracle.bin_vectors(g, B, q, mrl)
    short = int((rs.lens == q).sum())
    cap = 40_000 * (short + 1) + 200_000
    want = oracle.filter(oix, rs)
    for k in (1, 3, line, line + 1):
        sub = rs.subset(range(k))
        keep = want[0] < k
        assert_same(gpu_filter(ix, sub, cap=len(want[0]) + cap), tuple(x[keep] for x in want))
    plan = grim.grim_plan_create(ix, max_reads=line + 5, max_bases=len(rs.seq) + 64,
                                 max_e=mrl // 20, cap=len(want[0]) + cap)
    for k in (2, line + 1):
        sub = rs.subset(range(k))
        got = plan.run(**dev_reads(sub))
        keep = want[0] < k
        assert_same((got[0].cpu().numpy().view(np.uint32), got[1].cpu().numpy().view(np.uint32),
                     got[2].cpu().numpy()), tuple(x[keep] for x in want))
    plan.close()
    ix.close()


@pytest.mark.parametrize("q,layouts", [(4, 1), (5, 7), (5, 1), (6, 7)])
@pytest.mark.parametrize("n", [255, 256, 1025, 2500])
def test_mixed_batches_in_lockstep(q, layouts, n):
    """Mixed batches around the size from which they are sorted and run in
    lockstep, and around the sort's blocks of 1024 reads: reads of one token up
    to 255, budgets from 0 to T <= 0, non-bases, a repeat family that leaves
    more live words than a gather takes, a ragged last tile; the plain call, a
    plan, and output capacities that leave no room for the order."""
    from paper_1708_04329_gb300 import grim, synth

    rng = np.random.default_rng(n + q)
    g = synth.human_genome(400_000, seed=q)
    g[100_000:160_000] = np.resize(g[1000:1400], 60_000)
    rs = synth.reads(g, n, seed=n, lengths=(q, 40, 100, 254 + q), probs=(0.02, 0.28, 0.4, 0.3),
                     e_frac=(6, 100), max_edits=None)
    rs.e[rng.integers(0, n, 3)] = 200
    rs.e[rs.lens == q] = 0
    for r in rng.integers(0, n, 5):
        rs.seq[int(rs.offsets[r])] = ord("N")
    ix = build(g, 150, q, 254 + q, layouts)
    want = oracle.filter(oracle.bin_vectors(g, 150, q, 254 + q), rs)
    assert_same(gpu_filter(ix, rs, cap=len(want[0])), want)
    with pytest.raises(grim.GrimError):
        grim.grim_filter(ix, **dev_reads(rs), cap=10, retry=False)
    plan = grim.grim_plan_create(ix, max_reads=n + 3, max_bases=len(rs.seq), max_e=200,
                                 cap=len(want[0]) + 5)
    got = plan.run(**dev_reads(rs))
    assert_same((got[0].cpu().numpy().view(np.uint32), got[1].cpu().numpy().view(np.uint32),
                 got[2].cpu().numpy()), want)
    plan.close()
    ix.close()


@pytest.mark.parametrize("n", [4096 * 2 + 1, 4096 * 256, 4096 * 256 + 1])
def test_radix_sort_block_counts(n):
    """Pass lists of two and of 256 sort blocks and one record more (the scan
    of a digit's row takes a second step): every listed bin passes (T <= 0)."""
    rng = np.random.default_rng(n)
    g = rng.choice(np.frombuffer(b"ACGT", np.uint8), 30_000)
    nr = 300
    rs = Reads([g[p:p + 30].tobytes().decode() for p in rng.integers(0, 29_000, nr)], [15] * nr)
    cand = rng.integers(0, 600, n).astype(np.int32)
    off = np.sort(rng.integers(0, n + 1, nr + 1)).astype(np.uint64)
    off[0], off[-1] = 0, n
    ix = build(g, 50, 5, 30, layouts=2)
    r, b, _ = gpu_filter(ix, rs, off, cand, cap=n)
    assert np.array_equal(b.view(np.int32), cand)
    assert np.array_equal(r, np.repeat(np.arange(nr), np.diff(off.astype(np.int64))))
    ix.close()


@pytest.mark.parametrize("q,n,tail", [(4, 300, 1), (4, 70, 1025), (3, 257, 3 * 1024), (2, 300, 4095)])
def test_wide_tiles_of_small_q(q, n, tail):
    """q <= 4 with tiles enough for every SM: 4096-bin tiles, the last of them
    cut by the table's rows (which end on 1024 bins), mixed and uniform reads,
    non-bases, T <= 0; records and counts alone."""
    from paper_1708_04329_gb300 import grim, synth

    B = 9
    g = synth.genome(B * (4096 * 160 + tail), seed=q)
    rs = synth.reads(g, n, seed=n, lengths=(40, 60) if n > 70 else (40,),
                     probs=(0.5, 0.5) if n > 70 else (1.0,), e=1, max_edits=1)
    rs.seq[int(rs.offsets[3]) + 7] = ord("N")
    if n > 70:
        rs.e[5] = 60
    ix = build(g, B, q, 60, layouts=1)
    want = oracle.filter(oracle.bin_vectors(g, B, q, 60), rs)
    assert_same(gpu_filter(ix, rs, cap=len(want[0])), want)
    assert grim.grim_filter_count(ix, **dev_reads(rs)) == len(want[0])
    ix.close()
