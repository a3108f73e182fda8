"""Calls that give the same bits in every run: the strengths at every size, and the
gradients of the sizes whose sums go in a fixed order (up to 256 panels in the mixed
path, up to 64 in the plain FP64 one)."""
import numpy as np
import pytest

from paper_1511_02166_gb300 import inputs
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu

REPEATS = 12


def _batch(sizes, batch, mode="mixed", **kw):
    from paper_1511_02166_gb300.solver import PanelBatch
    rng = np.random.default_rng(batch + sum(sizes))
    base = [inputs.naca4(rng.uniform(0.01, 0.06), rng.uniform(0.2, 0.6), rng.uniform(0.08, 0.18),
                         int(n)) for n in sizes]
    pop = inputs.pack([base[b % len(base)] for b in range(batch)],
                      np.radians(rng.uniform(-4.0, 10.0, batch)))
    return pop, PanelBatch(pop.nodes, pop.offsets, pop.alpha, mode=mode, bucket_width=None, **kw)


def _same_every_time(call):
    first = [t.clone() for t in call()]
    for _ in range(REPEATS):
        for a, b in zip(first, call()):
            assert a.isfinite().all()
            assert np.array_equal(a.cpu().numpy().view(np.uint64), b.cpu().numpy().view(np.uint64))


@pytest.mark.parametrize("sizes,batch", [((160,), 1), ((100,), 64), ((256, 255, 225), 18),
                                         ((200,), 100), ((3, 31, 32, 33), 60), ((128,), 300)])
def test_mixed_gradients_repeat(sizes, batch):
    import torch
    need_gpu()
    pop, pb = _batch(sizes, batch)

    def step():
        pb.run(with_grad=True)
        return pb.u, pb.lam, pb.grad

    _same_every_time(step)
    w = torch.as_tensor(np.random.default_rng(1).normal(size=pb.total_nodes))
    _same_every_time(lambda: [pb.vjp(w_cp=w)])


@pytest.mark.parametrize("sizes,batch", [((64,), 1), ((40,), 64), ((3, 31, 32, 63, 64), 35),
                                         ((62,), 400), ((64, 12), 700)])
def test_fp64_gradients_repeat(sizes, batch):
    need_gpu()
    pop, pb = _batch(sizes, batch, mode="fp64")

    def step():
        pb.run(with_grad=True)
        return pb.u, pb.lam, pb.grad

    _same_every_time(step)


@pytest.mark.parametrize("sizes,batch", [((300, 290), 6), ((700, 400), 20), ((1100,), 3)])
def test_strengths_of_cluster_refinements_repeat(sizes, batch):
    need_gpu()
    pop, pb = _batch(sizes, batch)

    def step():
        pb.run(with_grad=True)
        return pb.u, pb.lam

    _same_every_time(step)


def test_gradient_refined_generations_repeat():
    need_gpu()
    from paper_1511_02166_gb300.ga import GeneticOptimizer
    out = []
    for _ in range(4):
        ga = GeneticOptimizer(32, 120, 0.05, seed=5, fitness="cl")
        ga.run(3, refine_lr=1e-3)
        out.append(ga.genome.cpu().numpy().copy())
    for g in out[1:]:
        assert np.array_equal(out[0].view(np.uint64), g.view(np.uint64))


@pytest.mark.parametrize("n,batch", [(3, 1), (33, 100), (100, 64), (128, 40), (129, 64), (160, 19),
                                     (200, 100), (256, 20), (255, 130)])
def test_small_batch_gradients_match_the_per_airfoil_kernel(n, batch):
    """The block shapes of a small batch against one block per airfoil (a batch that
    fills the chip): the same double-float sums in another order."""
    need_gpu()
    pop, pb = _batch((n, max(3, n - 1), max(3, n // 2)), batch)
    k = 1216 // batch + 1
    many_pop = inputs.pack([pop.airfoil(b) for b in range(batch)] * k, np.tile(pop.alpha, k))
    from paper_1511_02166_gb300.solver import PanelBatch
    many = PanelBatch(many_pop.nodes, many_pop.offsets, many_pop.alpha, bucket_width=None)
    grads = []
    for p in (pb, many):
        p.run(with_grad=True)
        assert int(p.info.abs().max()) == 0
        grads.append(p.grad.cpu().numpy()[:len(pop.nodes)])
    for b in range(batch):
        a, c = (g[pop.offsets[b]:pop.offsets[b + 1]] for g in grads)
        assert np.max(np.abs(a - c)) <= 1e-11 * np.max(np.abs(c))
