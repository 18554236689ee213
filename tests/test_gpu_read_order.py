"""The order in which the all-bins sweep takes the reads of a batch."""
import pytest

import oracle
from tests.gpu_helpers import assert_same, build, dev_reads, gpu_filter

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _mixed(g, q, n):
    from paper_1708_04329_gb300 import synth

    return synth.reads(g, n, seed=n + q, lengths=(60, 100, 150), probs=(0.4, 0.4, 0.2),
                       e_frac=(5, 100), max_edits=None)


@pytest.mark.parametrize("q,layouts", [(5, 7), (5, 1), (6, 7)])
def test_warp_switch_sorts_a_mixed_batch(q, layouts):
    """Set or automatic, the warp switch takes a mixed batch of 256 reads and more
    in sorted order, the group switch never; the pass lists are the same."""
    from paper_1708_04329_gb300 import grim, synth

    g = synth.genome(300_000, seed=q)
    rs = _mixed(g, q, 300)
    ix = build(g, 150, q, 150, layouts)
    want = oracle.filter(oracle.bin_vectors(g, 150, q, 150), rs)
    for switch, sorts in ((0, True), (grim.GRIM_SWITCH_WARP, True), (grim.GRIM_SWITCH_GROUP, False)):
        grim.grim_index_set_shape(ix, read_switch=switch)
        for k in (300, 255):
            sub = rs.subset(range(k))
            grim.grim_profile(True)
            got = gpu_filter(ix, sub, cap=len(want[0]) + 2000)
            assert ("order" in grim.grim_profile_get()) == (sorts and k >= 256)
            grim.grim_profile(False)
            assert_same(got, tuple(x[want[0] < k] for x in want))
        plan = grim.grim_plan_create(ix, max_reads=300, max_bases=len(rs.seq), max_e=10,
                                     cap=len(want[0]) + 5)
        got = plan.run(**dev_reads(rs))
        assert_same(tuple(x.cpu().numpy().view(w.dtype) for x, w in zip(got, want)), want)
        plan.close()
    ix.close()


@pytest.mark.parametrize("q,layouts", [(4, 1), (5, 7), (5, 1), (6, 1)])
@pytest.mark.parametrize("n", [255, 256, 1025])
def test_mixed_batches_without_room(q, layouts, n):
    """Calls whose output holds too little, or nothing, still count every passing
    pair, on indexes whose workspace has room for the order and on those whose
    record buffers would have to hold it."""
    from paper_1708_04329_gb300 import grim, synth

    g = synth.genome(200_000, seed=q + n)
    rs = _mixed(g, q, n)
    ix = build(g, 150, q, 150, layouts)
    want = oracle.filter(oracle.bin_vectors(g, 150, q, 150), rs)
    assert grim.grim_filter_count(ix, **dev_reads(rs)) == len(want[0]) > 10
    with pytest.raises(grim.GrimError) as ei:
        grim.grim_filter(ix, **dev_reads(rs), cap=10, retry=False)
    assert ei.value.code == grim.GRIM_E_OVERFLOW and ei.value.n_out == len(want[0])
    assert_same(gpu_filter(ix, rs, cap=10), want)
    ix.close()
