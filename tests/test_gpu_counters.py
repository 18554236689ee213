"""The work counters of grim_last_filter_stats."""
import pytest

from tests.gpu_helpers import build, gpu_filter

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("q,tile", [(5, 1024), (6, 256)])
@pytest.mark.parametrize("n", [1, 5, 300])
def test_tokens_are_counted_by_the_tables_tiles(q, tile, n):
    """A tile is left no sooner than D' + 1 tokens missed from it and no later
    than the read's end, in blocks of 16, whichever kernel sweeps it: batches of
    a few reads (1 and 5 against a table of 64 MB and more) and larger ones."""
    from paper_1708_04329_gb300 import grim, synth

    bins = 600_000 if q == 5 else 150_000  # 4^q rows of at least 64 MB together
    g = synth.genome(60 * bins, seed=q)
    ix = build(g, 60, q, 60, layouts=1)
    assert ix.desc.token_major_bytes >= 64 << 20
    rs = synth.reads(g, n, seed=n, lengths=(60,), e=5, max_edits=3)
    gpu_filter(ix, rs, cap=1_000_000)
    st = grim.grim_last_filter_stats()
    tiles = n * (ix.desc.num_bins_pad // tile)
    ntok, d = 60 - q + 1, 5 * q
    assert tiles * 16 * ((d + 1 + 15) // 16) <= st["tokens_executed"]
    assert st["tokens_executed"] <= tiles * 16 * ((ntok + 15) // 16)
    if n < 300:
        assert st["bit_tests_executed"] == st["tokens_executed"] * tile
    ix.close()
