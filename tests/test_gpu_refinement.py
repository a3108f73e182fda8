"""The refinement's stopping rule and its limits, in every form of the kernel."""
import numpy as np
import pytest

from paper_1511_02166_gb300 import binding as bd
from paper_1511_02166_gb300 import inputs
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


def _airfoils(sizes, seed=3):
    rng = np.random.default_rng(seed)
    return inputs.pack([inputs.naca4(rng.uniform(0.01, 0.06), rng.uniform(0.2, 0.6),
                                     rng.uniform(0.08, 0.18), int(n)) for n in sizes],
                       np.radians(rng.uniform(-4.0, 10.0, len(sizes))))


# (sizes, shape): one block with its vectors in shared memory, the same of more than
# 287 panels, and a cluster of blocks per airfoil
FORMS = [((40, 31), 0), ((250, 200), 0), ((300, 310), 4), ((300, 310), 0), ((700,), 0)]


@pytest.mark.parametrize("sizes,shape", FORMS)
def test_stopping_rule_takes_tolerances_beyond_float32(sizes, shape):
    """A zero right-hand side has the zero solution, converged under any tolerance:
    0 <= tol * 0 also for a tolerance that float32 cannot hold."""
    need_gpu()
    from paper_1511_02166_gb300.solver import PanelBatch
    pop = _airfoils(sizes)
    pb = PanelBatch(pop.nodes, pop.offsets, pop.alpha, vinf=np.zeros(len(sizes)), tol=1e39,
                    bucket_width=None)
    pb.ir_shape = [shape]
    pb.assemble()
    pb.solve()
    assert pb.info.cpu().tolist() == [0] * len(sizes)
    assert float(pb.u.abs().max()) == 0.0
    assert pb.iters.cpu().tolist() == [2] * len(sizes)  # the first iteration that tests


def _both_systems(pop, **set_):
    from paper_1511_02166_gb300.solver import PanelBatch
    pb = PanelBatch(pop.nodes, pop.offsets, pop.alpha, bucket_width=None,
                    **{k: v for k, v in set_.items() if k == "max_iter"})
    for name in ("ir_shape", "inverse"):
        if name in set_:
            setattr(pb, name, [set_[name]])
    pb.run(with_grad=True)
    return pb


def _kernel_names(call):
    import torch
    from torch.profiler import ProfilerActivity, profile
    for _ in range(3):  # (the first session of a process may come up empty)
        torch.cuda.synchronize()
        with profile(activities=[ProfilerActivity.CUDA]) as prof:
            call()
            torch.cuda.synchronize()
        names = " ".join(e.key for e in prof.key_averages())
        if "panel::" in names:
            return names
    return None  # no profiler here


@pytest.mark.parametrize("n", [60, 130, 260, 287])
@pytest.mark.parametrize("copies", [1, 8, 15])
def test_cluster_refinement_with_inverses(n, copies):
    """Gauss-Jordan inverses in a launch that an airfoil of more than 400 panels takes
    to clusters of 8, 4 or 2 blocks: both systems against the LU's."""
    need_gpu()
    base = _airfoils((n, n - 1, 50, 420), seed=n)
    pop = inputs.pack([base.airfoil(b) for b in range(4)] * copies, np.tile(base.alpha, copies))
    lu, inv = _both_systems(pop, inverse=False), _both_systems(pop, inverse=True)
    names = _kernel_names(lambda: inv.solve(with_adjoint=True, stage="refine"))
    assert names is None or "k_ir_cluster" in names
    assert int(lu.info.abs().max()) == 0 and int(inv.info.abs().max()) == 0
    # each ends within the refinement's 1e-12 of the same solution
    for a, c, tol in ((lu.u, inv.u, 1e-11), (lu.lam, inv.lam, 1e-11), (lu.grad, inv.grad, 1e-10)):
        assert float((a - c).abs().max()) <= tol * float(a.abs().max())


@pytest.mark.parametrize("sizes,shape", FORMS)
@pytest.mark.parametrize("max_iter", [0, 1])
def test_refinement_that_runs_out_of_steps(sizes, shape, max_iter):
    """No convergence is reported after max_iter steps, and no forces or gradients."""
    need_gpu()
    pb = _both_systems(_airfoils(sizes), ir_shape=shape, max_iter=max_iter)
    assert pb.info.cpu().tolist() == [bd.INFO_NOCONV] * len(sizes)
    assert pb.iters.cpu().tolist() == [max_iter] * len(sizes)
    assert pb.u.isfinite().all() and pb.lam.isfinite().all()
    assert pb.grad.isnan().all() and pb.cl.isnan().all()
