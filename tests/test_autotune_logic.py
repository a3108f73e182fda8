"""The autotuner's search and cache without a GPU: timings and device are stand-ins."""
import types

import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_1511_02166_gb300 import binding as bd  # noqa: E402
from paper_1511_02166_gb300 import build, solver  # noqa: E402


@pytest.fixture
def tuned(tmp_path, monkeypatch):
    """tuned(count, n) -> (choices, calls timed) of a batch of equal airfoils, every
    candidate taking the same time."""
    monkeypatch.setenv("PANEL_AUTOTUNE_CACHE", str(tmp_path / "tune.json"))
    monkeypatch.setattr(torch.cuda, "get_device_name", lambda d=None: "device")
    monkeypatch.setattr(torch.cuda, "get_device_properties",
                        lambda d=None: types.SimpleNamespace(multi_processor_count=152))
    monkeypatch.setattr(torch.cuda, "synchronize", lambda d=None: None)

    def run(count, n):
        pb = solver.PanelBatch.__new__(solver.PanelBatch)
        pb.flags, pb.device, pb.B = bd.PANEL_MIXED, "cuda", count
        pb.offsets_h = np.arange(count + 1) * n
        pb.buckets = [(0, count, n)]
        pb.bucket_width = None
        pb.order = torch.arange(count)
        pb.info = torch.zeros(count, dtype=torch.int32)
        pb._reset_tuning()
        pb.assemble = lambda: None
        timed = []
        pb._time = lambda fn, reps: timed.append(fn) or 1.0
        return pb, pb.autotune(reps=1), timed

    return run


@pytest.mark.parametrize("n", [10, 64, 100, 160, 200, 221, 222, 287, 288, 639, 640, 2048])
@pytest.mark.parametrize("count", [1, 152, 153, 4096])
def test_without_a_faster_candidate_the_librarys_choice_stays(tuned, count, n):
    pb, chosen, timed = tuned(count, n)
    assert len(timed) == 7 + 6 * len(solver.solve_candidates(n))
    assert (pb.inverse, pb.ir_shape, pb.lu_kind, pb.rounds) == ([False], [0], [0], [0])


def test_choices_are_kept_per_exact_small_batch_and_per_library(tuned, monkeypatch):
    _, first, timed = tuned(7, 600)
    assert len(timed) > 0 and all(build.source_key() in k for k in first)
    _, again, timed = tuned(7, 600)
    assert again == first and not timed
    # another count below eight airfoils per multiprocessor is another choice ...
    for count in (1, 8, 150, 152, 153, 1215):
        _, other, timed = tuned(count, 600)
        assert len(timed) > 0 and not set(other) & set(first)
    # ... above they share one, and other sources share none
    _, large, _ = tuned(1216, 600)
    _, larger, timed = tuned(10000, 600)
    assert larger == large and not timed
    monkeypatch.setattr(build, "source_key", lambda: "another")
    _, other, timed = tuned(7, 600)
    assert len(timed) > 0 and not set(other) & set(first)


def test_source_key_follows_the_sources(tmp_path, monkeypatch):
    src = tmp_path / "a.cu"
    src.write_text("one")
    monkeypatch.setattr(build, "_deps", lambda: [str(src)])
    one = build.source_key()
    src.write_text("two")
    assert build.source_key() != one and len(one) == 12
