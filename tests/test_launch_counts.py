"""Kernel launches of a step: the library's own count, by the rules its launches go by,
and what a profiler sees."""
import numpy as np
import pytest

from paper_1511_02166_gb300 import binding as bd
from paper_1511_02166_gb300 import inputs
from tests.gpu_util import need_gpu

MIXED, FP64 = bd.PANEL_MIXED, bd.PANEL_FP64
SMS = 152

COUNTS = [
    # the assembly: one block per airfoil, or a preparing launch and the pairs
    (bd.CALL_ASSEMBLE, 4096, 300, FP64, 1),
    (bd.CALL_ASSEMBLE, 1, 64, MIXED, 1),
    (bd.CALL_ASSEMBLE, 1, 160, MIXED, 2),
    (bd.CALL_ASSEMBLE, 50, 128, MIXED, 2),
    (bd.CALL_ASSEMBLE, 51, 128, MIXED, 1),
    (bd.CALL_ASSEMBLE, SMS + 1, 224, MIXED, 1),
    (bd.CALL_ASSEMBLE, SMS + 1, 225, MIXED, 2),
    (bd.CALL_ASSEMBLE, 114, 144, MIXED, 2),
    (bd.CALL_ASSEMBLE, 115, 144, MIXED, 1),
    (bd.CALL_ASSEMBLE, 115, 145, MIXED, 2),
    (bd.CALL_ASSEMBLE, 1, 160, MIXED | bd.PANEL_TUNE_ROUNDS(1), 1),
    (bd.CALL_ASSEMBLE, 4096, 200, MIXED | bd.PANEL_TUNE_ROUNDS(6), 2),
    # factor and refinement
    (bd.CALL_SOLVE, 4096, 300, FP64, 1),
    (bd.CALL_SOLVE, 1, 40, MIXED, 2),
    (bd.CALL_SOLVE, 4096, 100, MIXED, 2),
    (bd.CALL_SOLVE, 1, 639, MIXED, 2),
    (bd.CALL_SOLVE, 1, 300, MIXED | bd.PANEL_TUNE_LU(2), 3),
    (bd.CALL_SOLVE, 1, 100, MIXED | bd.PANEL_INVERSE, 2),
    (bd.CALL_SOLVE, 1, 250, MIXED | bd.PANEL_INVERSE, 3),
    (bd.CALL_SOLVE, 1, 300, MIXED | bd.PANEL_INVERSE, 4),
    # 1025 unknowns, T = 9: copy, 9 diagonal blocks, 8 solves and 8 updates, the U tiles,
    # the finishing pass, the smaller airfoils' LU, the refinement
    (bd.CALL_SOLVE, 1, 1024, MIXED, 1 + 9 + 16 + 1 + 1 + 1 + 1),
    (bd.CALL_SOLVE, 1, 100, MIXED | bd.PANEL_FACTOR_ONLY, 1),
    (bd.CALL_SOLVE, 1, 1024, MIXED | bd.PANEL_REUSE_FACTOR, 1),
    # the adjoint: sums in a fixed order, or the terms without pair sums first
    (bd.CALL_ADJOINT, 1, 256, MIXED, 1),
    (bd.CALL_ADJOINT, 4096, 257, MIXED, 2),
    (bd.CALL_ADJOINT, 4096, 64, FP64, 1),
    (bd.CALL_ADJOINT, 1, 65, FP64, 2),
]


@pytest.mark.parametrize("call,B,n,flags,count", COUNTS)
def test_library_counts_its_launches(call, B, n, flags, count):
    assert bd.panel_launches(call, B, n, flags, SMS) == count


def test_launch_counts_refuse_invalid_arguments():
    for args in [(3, 1, 10, MIXED, SMS), (0, -1, 10, MIXED, SMS), (0, 1, 2, MIXED, SMS),
                 (0, 1, 2049, MIXED, SMS), (0, 1, 10, 0, SMS), (0, 1, 10, MIXED, 0)]:
        with pytest.raises(bd.PanelError):
            bd.panel_launches(*args)
    assert bd.panel_launches(bd.CALL_SOLVE, 0, 10, MIXED, SMS) == 0


def _kernels(call):
    """Launches of the library's kernels by one call (the first session of a process may
    come up empty: it is repeated on a call of its own)."""
    import torch
    from torch.profiler import ProfilerActivity, profile
    for _ in range(3):
        torch.cuda.synchronize()
        with profile(activities=[ProfilerActivity.CUDA]) as prof:
            call()
            torch.cuda.synchronize()
        seen = sum(e.count for e in prof.key_averages() if "panel::" in e.key)
        if seen:
            return seen
    pytest.skip("the profiler sees no kernels here")


@pytest.mark.gpu
@pytest.mark.parametrize("mode,sizes,batch", [
    ("fp64", (100, 64), 5), ("fp64", (64,), 5), ("fp64", (200,), 160), ("mixed", (160,), 1),
    ("mixed", (64, 40), 3), ("mixed", (128, 100), 200), ("mixed", (200,), 160),
    ("mixed", (250, 300), 40), ("mixed", (700, 40), 4), ("mixed", (40, 90, 200), 1500)])
@pytest.mark.parametrize("with_grad", [False, True])
def test_steps_launch_as_many_kernels_as_they_count(mode, sizes, batch, with_grad):
    need_gpu()
    from paper_1511_02166_gb300.solver import PanelBatch
    base = [inputs.naca4(0.02, 0.4, 0.12, n) for n in sizes]
    pop = inputs.pack([base[b % len(base)] for b in range(batch)], np.full(batch, 0.05))
    pb = PanelBatch(pop.nodes, pop.offsets, pop.alpha, mode=mode, bucket_width=64, bucket_min=100)
    inverses = (False, True) if mode == "mixed" else (False,)
    for inverse in inverses:
        pb.inverse = [inverse] * len(pb.buckets)
        pb.run(with_grad=with_grad)
        assert _kernels(lambda: pb.run(with_grad=with_grad)) == pb.launches_per_step(with_grad=with_grad)
