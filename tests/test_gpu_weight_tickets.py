"""Weight builds of few stencils and of counts around the number of resident teams:
each row has the bits it has in a build of all rows (a stencil's system does not
depend on the team that solves it)."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rb():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2502_12878_gb300 import build as nvbuild
    nvbuild.build()
    import paper_2502_12878_gb300 as m
    m.lib()
    return m


@pytest.mark.parametrize("d,Kg,m,n", [(2, 80, 2, 12), (2, 80, 4, 30), (2, 60, 6, 56), (3, 14, 4, 70)])
def test_counts(rb, d, Kg, m, n):
    xyz, bnd = rb.rbffd_nodes(d, 0, Kg, 0.3, 2)
    idx = rb.rbffd_knn(xyz, rb.rbffd_interior(bnd), n)
    w, _ = rb.rbffd_weights(xyz, idx, m)
    for k in (1, 2, 7, 151, 152, 153, 303, 841, 1975, 1976, 1977, 2432, 3953, idx.shape[0] - 1):
        if k < idx.shape[0]:
            assert torch.equal(rb.rbffd_weights(xyz, idx[-k:].contiguous(), m)[0], w[-k:])


@pytest.mark.parametrize("d,Kg,m,n", [(2, 200, 4, 30), (2, 200, 4, 31), (2, 140, 2, 13),
                                      (2, 70, 6, 57), (3, 16, 4, 71)])
def test_long_and_short_builds(rb, d, Kg, m, n):
    """Builds on either side of the rounds of stencils at which teams begin to draw tickets ahead
    or to draw them at all, one call and several calls in one launch."""
    xyz, bnd = rb.rbffd_nodes(d, 0, Kg, 0.3, 2)
    idx = rb.rbffd_knn(xyz, rb.rbffd_interior(bnd), n)
    w, _ = rb.rbffd_weights(xyz, idx, m)
    cuts = [0, 1, 33, 900, 2001, idx.shape[0]]
    parts = [idx[a:b].contiguous() for a, b in zip(cuts, cuts[1:])]
    assert torch.equal(torch.cat([rb.rbffd_weights(xyz, p, m)[0] for p in parts]), w)
    both = rb.rbffd_weights_batch([xyz] * len(parts), parts, [m] * len(parts))
    assert torch.equal(torch.cat([x for x, _ in both]), w)
