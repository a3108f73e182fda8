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
