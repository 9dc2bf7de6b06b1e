"""Contexts and calls that are at work at the same time do not change one another's launches:
a kernel's limit of dynamic shared memory belongs to the process, whichever size asked for it."""
import threading

import pytest

from paper_1203_6402_gb300 import datagen

torch = pytest.importorskip("torch")


@pytest.mark.gpu
def test_a_smaller_context_leaves_a_larger_one_alone():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1203_6402_gb300 import kmpar as km
    X = torch.from_numpy(datagen.uniform_box(120_000, 2, seed=1)).cuda()
    a = km.KMeansPar(X, 40_000, 12_000.0, 1, 7)   # a sort of 16,384 draws, counters of 40,000 labels
    b = km.KMeansPar(X, 13_000, 20.0, 1, 7)
    a.round(1, sync=True)
    assert a.lloyd(X[:40_000].clone(), 1)["iters"] == 1
    assert b.lloyd(X[:13_000].clone(), 1)["iters"] == 1
    a.close()
    b.close()


def _in_turn(jobs, times):
    """Each job `times` times on a thread of its own; what they raised."""
    start, bad = threading.Barrier(len(jobs)), []

    def work(job):
        try:
            start.wait()
            for _ in range(times):
                job()
        except Exception as e:
            bad.append(e)

    threads = [threading.Thread(target=work, args=(j,)) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    return bad


@pytest.mark.gpu
def test_costs_of_two_dimensions_on_two_threads():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1203_6402_gb300 import kmpar as km
    jobs = []
    for d in (50, 96):
        X = torch.from_numpy(datagen.gauss_mixture(41_000, d, 20, 10.0, seed=d)).cuda()
        s = torch.cuda.Stream()
        s.wait_stream(torch.cuda.current_stream())
        want = km.kmpar_cost(X.data_ptr(), len(X), d, X.data_ptr(), 40)

        def job(X=X, d=d, s=s, want=want):
            assert km.kmpar_cost(X.data_ptr(), len(X), d, X.data_ptr(), 40, stream=s.cuda_stream) == want

        jobs.append(job)
    torch.cuda.synchronize()
    assert not _in_turn(jobs, 4000)
