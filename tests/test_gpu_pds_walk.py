"""The 2D walk's single launch where its branches differ, against the oracle's sequential walk
(bit for bit, as every placement test): one and many candidates a parent (64: dozens of
conflicts each, past what a warp collects in shared memory), a small zeta, the smallest sets,
and generations whose lists do not fit shared memory."""
import numpy as np
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


@pytest.mark.parametrize("shape,Kg,seed,K,zeta", [
    (0, 2, 1, 15, 1 - 1e-10),
    (0, 3, 2, 1, 1.0),
    (0, 200, 3, 1, 1 - 1e-10),
    (0, 150, 4, 6, 1.0),                # siblings at distance h of each other: FP64 decides
    (0, 60, 5, 64, 1 - 1e-10),
    (1, 40, 6, 64, 0.3),
    (0, 1400, 7, 15, 1 - 1e-10),        # 15,000 candidates a generation
    (0, 500, 8, 64, 1 - 1e-10),
])
def test_walk_equals_the_sequential_one(rb, orc, shape, Kg, seed, K, zeta):
    xyz, bnd, rounds = rb.rbffd_nodes_pds(shape, Kg, seed, K=K, zeta=zeta)
    oxyz, obnd = orc.nodes_pds(shape, Kg, seed, K=K, zeta=zeta)
    assert xyz.shape == oxyz.shape
    assert np.array_equal(xyz.cpu().numpy(), oxyz) and np.array_equal(bnd.cpu().numpy(), obnd)
    assert rounds >= 1
