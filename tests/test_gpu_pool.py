"""The library's memory pool under several threads and streams at once: each thread computes
supports, weights, their application, a Poisson-disc fill and errors of its own node sets on its
own stream and gets what a single thread gets, bit for bit."""
import threading

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _work(rb, kg):
    xyz, bnd = rb.rbffd_nodes(2, 0, kg, 0.3, kg)
    inter = rb.rbffd_interior(bnd)
    idx = rb.rbffd_knn(xyz, inter, 12)
    w, _ = rb.rbffd_weights(xyz, idx, 2)
    u = xyz.square().sum(0)
    fill, fbnd, _ = rb.rbffd_nodes_pds(0, kg, kg)
    return [idx, w, rb.rbffd_apply(w, idx, u), fill, fbnd, torch.tensor(rb.rbffd_error(u, u * 2))]


def test_threads_and_streams_share_the_pool():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2502_12878_gb300 import build as nvbuild
    nvbuild.build()
    import paper_2502_12878_gb300 as rb
    sizes = [20, 45, 70, 95]
    want = {kg: _work(rb, kg) for kg in sizes}
    torch.cuda.synchronize()
    wrong = []

    def go(kg):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(10):
                    got = _work(rb, kg)
                    torch.cuda.current_stream().synchronize()
                    wrong.extend((kg, i) for i, (a, b) in enumerate(zip(got, want[kg]))
                                 if not torch.equal(a, b))
        except Exception as e:   # a thread's failure is the test's
            wrong.append((kg, repr(e)))

    threads = [threading.Thread(target=go, args=(kg,)) for kg in sizes]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong, wrong
