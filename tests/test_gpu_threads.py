"""Calls from several host threads at once, whose kernels ask for different
amounts of shared memory: one thread's call must not take away what another's is
about to launch with."""
import threading

import numpy as np
import pytest

from tests.gpu_helpers import dev_reads

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _together(jobs):
    """Run the jobs in threads of their own, on streams of their own."""
    failed, start = [], threading.Barrier(len(jobs))

    def work(job):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                start.wait()
                for _ in range(400):
                    job()
        except Exception as e:  # noqa: BLE001 -- whatever it is, the test reports it
            failed.append(e)

    threads = [threading.Thread(target=work, args=(j,)) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed


@pytest.mark.parametrize("q,shapes", [(5, ((64, 100), (700, 100))), (6, ((50, 150), (1000, 150))),
                                      (4, ((50, 40), (50, 41)))])
def test_builds_of_different_shapes_at_once(q, shapes):
    from paper_1708_04329_gb300 import grim

    rng = np.random.default_rng(q)
    ref = torch.from_numpy(rng.choice(np.frombuffer(b"ACGT", np.uint8), 20_000)).cuda()
    torch.cuda.synchronize()
    qs = (q, 3) if q == 4 else (q, q)  # q = 4 and 3 share a kernel too
    _together([lambda B=B, m=m, k=k: grim.grim_build_ex(ref, B, k, m).close()
               for (B, m), k in zip(shapes, qs)])


def test_filters_of_different_indexes_at_once():
    from paper_1708_04329_gb300 import grim, synth

    g = synth.genome(20_000, seed=3)
    ref = torch.from_numpy(g).cuda()
    jobs = []
    for mrl in (60, 250):
        ix = grim.grim_build_ex(ref, 200, 5, mrl, grim.GRIM_LAYOUT_TOKEN_MAJOR)
        kw = dev_reads(synth.reads(g, 8, seed=4, lengths=(50,), e=2, max_edits=2))
        want = len(grim.grim_filter(ix, **kw)[0])

        def job(ix=ix, kw=kw, want=want):
            assert len(grim.grim_filter(ix, **kw)[0]) == want

        jobs.append(job)
    torch.cuda.synchronize()
    _together(jobs)
