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


def test_a_destroyed_plan_gives_its_memory_back_at_once():
    """What the pool keeps is bounded by 128 MB whatever the size of the plan that went, and a
    caller need not synchronise to get the rest."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2502_12878_gb300 as rb
    kg, n = 1000, 56
    N = (kg + 1) ** 2
    xyz, bnd = rb.rbffd_nodes(2, 0, kg, 0.3, 1)
    inter = rb.rbffd_interior(bnd)
    idx = inter[:, None].repeat(1, n)
    w = torch.zeros((inter.numel(), n), dtype=torch.float64, device="cuda")
    rb.Plan(xyz, bnd, inter, idx, w).destroy()
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    plan = rb.Plan(xyz, bnd, inter, idx, w)
    assert before - torch.cuda.mem_get_info()[0] > 600 << 20
    plan.destroy()
    assert torch.cuda.mem_get_info()[0] >= before - (160 << 20)
    assert N == xyz.shape[1]


def test_threads_make_and_destroy_plans():
    """Plans are arrays of the pool too: made, used and destroyed by several threads at once."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2502_12878_gb300 as rb

    def work(kg, flags):
        xyz, bnd = rb.rbffd_nodes(2, 0, kg, 0.3, kg)
        inter = rb.rbffd_interior(bnd)
        idx = rb.rbffd_knn(xyz, inter, 12)
        w, _ = rb.rbffd_weights(xyz, idx, 2)
        plan = rb.Plan(xyz, bnd, inter, idx, w, flags)
        out = plan.perm().tolist(), plan.stable_dt(xyz[0][inter.long()] + 0.1, 70)
        plan.destroy()
        return out

    jobs = [(20, 0), (45, 64), (70, 64), (95, 0), (33, 64), (120, 64)]
    want = {j: work(*j) for j in jobs}
    torch.cuda.synchronize()
    wrong = []

    def go(job):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                wrong.extend(job for _ in range(8) if work(*job) != want[job])
        except Exception as e:   # a thread's failure is the test's
            wrong.append((job, repr(e)))

    threads = [threading.Thread(target=go, args=(j,)) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong, wrong
