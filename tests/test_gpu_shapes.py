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


@pytest.mark.parametrize("n", [31, 222, 223, 255, 256, 286, 351, 380, 384, 480, 639])
def test_lu_through_l2_with_two_and_three_blocks_per_sm(n):
    """The L2-resident LU's two forms (by batch and shared memory) do the same
    operations; small batches are compared with the shared-memory form above."""
    need_gpu()
    import torch
    from paper_1511_02166_gb300.solver import PanelBatch
    base = _airfoils((n, max(3, n - 1)), seed=n)
    one, many = base, inputs.pack([base.airfoil(b) for b in range(2)] * 160,
                                  np.tile(base.alpha, 160))
    out = []
    for pop in (one, many):
        pb = PanelBatch(pop.nodes, pop.offsets, pop.alpha, bucket_width=None)
        pb.lu_kind = [1]
        pb.run(with_grad=False)
        assert int(pb.info.abs().max()) == 0
        m = n + 1
        A = (pb.A_hi[:m * m].double() + pb.A_lo[:m * m].double()).reshape(m, m)
        x = torch.linalg.solve(A, pb.rhs[:m])
        u = pb.u[:m].clone()
        # the refinement stops at 1e-12 of the largest strength; the 64-bit solve's
        # own error is cond(A) 2^-53 (up to ~1e4 here)
        assert float((u - x).abs().max()) <= 1e-11 * float(x.abs().max())
        out.append((pb.LU[:m * m].cpu().numpy().view(np.uint32), pb.piv[:m].cpu().numpy()))
    assert np.array_equal(out[0][0], out[1][0])
    assert np.array_equal(out[0][1], out[1][1])


@pytest.mark.parametrize("sizes", [(3, 70), (65, 96, 97), (127, 128, 129), (160,), (255, 257, 31),
                                   (15, 16, 17, 400), (1030, 640)])
@pytest.mark.parametrize("copies", [1, 40])
def test_assembly_kernels_give_the_same_matrix(sizes, copies):
    """The forms chosen by batch and size (split rows, tiles of 64 and 128 panels)
    against one block per airfoil: every entry by the same operations."""
    need_gpu()
    from paper_1511_02166_gb300.solver import PanelBatch
    base = _airfoils(sizes, seed=sum(sizes))
    pop = inputs.pack([base.airfoil(b) for b in range(len(sizes))] * copies,
                      np.tile(base.alpha, copies))
    out = []
    for rounds in (1, 0, 6):
        pb = PanelBatch(pop.nodes, pop.offsets, pop.alpha, bucket_width=None)
        for t in (pb.A_hi, pb.A_lo, pb.rhs):
            t.fill_(float("nan"))
        pb.rounds = [rounds]
        pb.assemble()
        assert int(pb.info.abs().max()) == 0
        out.append([t.cpu().numpy() for t in (pb.A_hi, pb.A_lo, pb.rhs)])
        assert all(np.isfinite(t).all() for t in out[-1])
    for other in out[1:]:
        assert np.array_equal(out[0][0].view(np.uint32), other[0].view(np.uint32))
        assert np.array_equal(out[0][1].view(np.uint32), other[1].view(np.uint32))
        assert np.max(np.abs(out[0][2] - other[2])) <= 1e-15


@pytest.mark.parametrize("n", [80, 300])
def test_assembly_of_a_small_batch_reports_bad_geometry(n):
    """The codes of the several-block forms: clockwise, zero panel, non-finite, good."""
    need_gpu()
    import torch
    from paper_1511_02166_gb300.solver import PanelBatch
    good = inputs.naca4(0.02, 0.4, 0.12, n)
    zero, nan = good.copy(), good.copy()
    zero[n - 1] = zero[0]
    nan[n // 2, 1] = np.nan
    pop = inputs.pack([good[::-1].copy(), zero, nan, good], [0.05] * 4)
    pb = PanelBatch(pop.nodes, pop.offsets, pop.alpha, bucket_width=None)
    pb.run(with_grad=True)
    torch.cuda.synchronize()
    assert pb.info.cpu().tolist() == [-2, -3, -4, 0]
    assert torch.isnan(pb.cl[:3]).all() and torch.isfinite(pb.cl[3])
    assert torch.isfinite(pb.grad[-n:]).all() and torch.isnan(pb.grad[:-n]).all()


@pytest.mark.parametrize("sizes", [(128,), (129, 200, 160), (287, 288), (300, 639, 640), (641, 767),
                                   (1024, 1040, 700, 40)])
@pytest.mark.parametrize("copies", [1, 12, 30])
def test_cluster_refinement_matches_the_one_block_refinement(sizes, copies):
    """A batch that fits the chip as clusters of 8, 4, 2 or 1 blocks against the
    explicit one-block shape: both end within the tolerance of the same solution
    (up to 700 panels far below it; the larger airfoils' conditioning is 1e9)."""
    need_gpu()
    import torch
    from paper_1511_02166_gb300.solver import PanelBatch
    base = _airfoils(sizes, seed=len(sizes) + sizes[0])
    pop = inputs.pack([base.airfoil(b) for b in range(len(sizes))] * copies,
                      np.tile(base.alpha, copies))
    out = []
    for shape in (4, 0):
        pb = PanelBatch(pop.nodes, pop.offsets, pop.alpha, bucket_width=None)
        pb.ir_shape = [shape]
        pb.run(with_grad=True)
        cl = pb.polar(torch.tensor([[0.0, 0.1]] * pop.batch))
        assert int(pb.info.abs().max()) == 0
        out.append([t.cpu().numpy() for t in (pb.u, pb.lam, cl)])
    for a, c in zip(out[0][:2], out[1][:2]):
        for b in range(pop.batch):
            o, n = pop.offsets[b] + b, pop.offsets[b + 1] - pop.offsets[b]
            tol = 1e-11 if n <= 700 else 1e-10
            assert np.max(np.abs(a[o:o + n + 1] - c[o:o + n + 1])) <= tol * np.max(np.abs(a[o:o + n + 1])), b
    assert np.max(np.abs(out[0][2] - out[1][2])) <= 1e-11


@pytest.mark.parametrize("n", [130, 260])
def test_cluster_refinement_with_the_inverse(n):
    """The Gauss-Jordan inverse through the cluster refinement."""
    need_gpu()
    from paper_1511_02166_gb300.solver import PanelBatch
    pop = _airfoils((n, n - 1, 50), seed=n)
    out = []
    for inverse in (False, True):
        pb = PanelBatch(pop.nodes, pop.offsets, pop.alpha, bucket_width=None)
        pb.inverse = [inverse]
        pb.run(with_grad=True)
        assert int(pb.info.abs().max()) == 0
        out.append((pb.u.cpu().numpy(), pb.grad.cpu().numpy()))
    assert np.max(np.abs(out[0][0] - out[1][0])) <= 1e-11 * np.max(np.abs(out[0][0]))
    assert np.max(np.abs(out[0][1] - out[1][1])) <= 1e-10 * np.max(np.abs(out[0][1]))


@pytest.mark.parametrize("n", [3, 30, 31, 32, 61, 62, 63, 64, 93, 127, 128, 158, 159, 160, 170])
def test_fp64_path_at_the_edges_of_its_tiles(n):
    """31-panel column blocks, row ranges, the matrix in shared memory or not: against
    the oracle, and the transposed solve of panel_adjoint against panel_solve's."""
    need_gpu()
    import oracle
    from paper_1511_02166_gb300.solver import PanelBatch
    pop = _airfoils((n, max(3, n - 1), max(3, n // 2)), seed=n)
    ref = oracle.evaluate_batch(pop.nodes, pop.offsets, pop.alpha)
    pb = PanelBatch(pop.nodes, pop.offsets, pop.alpha, mode="fp64", bucket_width=None)
    pb.run(with_grad=True)
    assert int(pb.info.abs().max()) == 0
    u, lam, g = (t.cpu().numpy() for t in (pb.u, pb.lam, pb.grad))
    assert np.max(np.abs(u - ref["u"])) <= 1e-10 * np.max(np.abs(ref["u"]))
    assert np.max(np.abs(pb.cl.cpu().numpy() - ref["cl"])) <= 1e-10
    assert np.max(np.abs(pb.cl_p.cpu().numpy() - ref["cl_p"])) <= 1e-10
    grad, _ = oracle.cl_gradient_batch(pop.nodes, pop.offsets, pop.alpha)
    assert np.max(np.abs(g - grad)) <= 1e-9 * np.max(np.abs(grad))
    pb.solve(with_adjoint=False)
    pb.adjoint()
    assert np.max(np.abs(pb.lam.cpu().numpy() - lam)) <= 1e-11 * np.max(np.abs(lam))


@pytest.mark.parametrize("batch", [1, 609])
@pytest.mark.parametrize("n", [3, 31, 33, 127, 129, 300])
def test_forces_by_one_and_by_four_warps(batch, n):
    """Cp, Cl and the pressure forces of both block shapes with vinf and chord given."""
    need_gpu()
    from paper_1511_02166_gb300.solver import PanelBatch
    pop = _airfoils((n,), seed=n)
    pop = inputs.pack([pop.airfoil(0)] * batch, np.tile(pop.alpha, batch))
    v, c = np.full(batch, 1.7), np.full(batch, 0.9)
    pb = PanelBatch(pop.nodes, pop.offsets, pop.alpha, vinf=v, chord=c, bucket_width=None)
    pb.run()
    x, a = pop.airfoil(batch - 1), pop.alpha[-1]
    g = pb.gamma(batch - 1).cpu().numpy()
    h = np.roll(x, -1, axis=0) - x
    cp = 1 - (g / 1.7)**2
    f = np.array([-(cp * h[:, 1]).sum(), (cp * h[:, 0]).sum()])
    tol = 1e-13 * (1 + np.abs(cp).sum())
    assert np.max(np.abs(pb.cp[-n:].cpu().numpy() - cp)) <= 1e-13 * np.max(np.abs(cp))
    assert abs(float(pb.cl[-1]) - 2 * (g * np.hypot(*h.T)).sum() / (1.7 * 0.9)) <= tol
    assert abs(float(pb.cl_p[-1]) - (-f[0] * np.sin(a) + f[1] * np.cos(a)) / 0.9) <= tol
    assert abs(float(pb.cd_p[-1]) - (f[0] * np.cos(a) + f[1] * np.sin(a)) / 0.9) <= tol
