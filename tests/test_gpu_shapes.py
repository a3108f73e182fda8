"""Launch shapes: the kernels a small batch takes against the ones a large batch
takes, at the edges of their tiles."""
import numpy as np
import pytest

from paper_1511_02166_gb300 import inputs
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


def _airfoils(sizes, seed=3):
    rng = np.random.default_rng(seed)
    return inputs.pack([inputs.naca4(rng.uniform(0.01, 0.06), rng.uniform(0.2, 0.6),
                                     rng.uniform(0.08, 0.18), int(n)) for n in sizes],
                       np.radians(rng.uniform(-4.0, 10.0, len(sizes))))


@pytest.mark.parametrize("sizes", [(3,), (31, 32, 33), (63, 64, 65), (127, 128, 129), (255, 256),
                                   (5, 200)])
def test_split_adjoint_of_a_small_batch_matches_the_per_airfoil_kernel(sizes):
    """A batch that fills the chip takes one block per airfoil, a small one the
    split contraction: the same sums in another order, each rounded to ~1e-13."""
    need_gpu()
    from paper_1511_02166_gb300.solver import PanelBatch
    small = _airfoils(sizes)
    copies = 1300
    many = inputs.pack([small.airfoil(b) for b in range(len(sizes))] * copies,
                       np.tile(small.alpha, copies))
    grads = []
    for pop in (small, many):
        pb = PanelBatch(pop.nodes, pop.offsets, pop.alpha, bucket_width=None)
        pb.run(with_grad=True)
        assert int(pb.info.abs().max()) == 0
        grads.append(pb.grad.cpu().numpy()[:len(small.nodes)])
    for b in range(len(sizes)):
        a, c = (g[small.offsets[b]:small.offsets[b + 1]] for g in grads)
        assert np.max(np.abs(a - c)) <= 1e-11 * np.max(np.abs(c))


@pytest.mark.parametrize("n", [3, 30, 31, 32, 62, 63, 64, 95, 126, 127, 128, 159, 191, 220, 221])
def test_lu_in_shared_memory_and_through_l2_agree(n):
    """Both one-block LUs do the same operations in the same order at every edge of
    their 32-column panels and of the shared-memory form's block sizes."""
    need_gpu()
    from paper_1511_02166_gb300.solver import PanelBatch
    pop = _airfoils((n, n, max(3, n - 1)), seed=n)
    out = []
    for kind in (1, 2):
        pb = PanelBatch(pop.nodes, pop.offsets, pop.alpha, bucket_width=None)
        pb.lu_kind = [kind]
        pb.assemble()
        pb.solve(stage="factor")
        assert int(pb.info.abs().max()) == 0
        out.append((pb.LU.cpu().numpy().view(np.uint32), pb.piv.cpu().numpy()))
    assert np.array_equal(out[0][0], out[1][0])
    assert np.array_equal(out[0][1], out[1][1])
