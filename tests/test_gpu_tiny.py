"""Airfoils so small that products of their lengths leave float32's range: the geometry
checks accept them, and their entries are NaN or finite, alike in every form of the
assembly, with none left as it was."""
import numpy as np
import pytest

from paper_1511_02166_gb300 import inputs
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("exponent", [0, -40, -60, -64, -70, -90])
@pytest.mark.parametrize("n", [20, 100, 300])
def test_tiny_airfoils_assemble_alike_in_every_form(exponent, n):
    need_gpu()
    from paper_1511_02166_gb300.solver import PanelBatch
    foil = inputs.naca4(0.02, 0.4, 0.12, n) * 2.0**exponent
    pop = inputs.pack([foil, foil], [0.05, 0.1])
    out = []
    for rounds in (1, 4, 0, 6):
        pb = PanelBatch(pop.nodes, pop.offsets, pop.alpha, bucket_width=None)
        pb.A_hi.fill_(7.0)
        pb.A_lo.fill_(7.0)
        pb.rounds = [rounds]
        pb.assemble()
        assert pb.info.cpu().tolist() == [0, 0]
        out.append((pb.A_hi.cpu().numpy(), pb.A_lo.cpu().numpy()))
    for hi, lo in out:
        assert not (hi == 7.0).any() and not (lo == 7.0).any()
        assert np.array_equal(out[0][0], hi, equal_nan=True)
        assert np.array_equal(out[0][1], lo, equal_nan=True)
