"""The wavefront engine under the calls whose other tests run the merging engine
(contexts with default settings): the full batches against the oracle's hashes,
the segmented host pipeline with and without planning, planning inside recon_batch,
calls back to back with a graph replay. They are the same test functions, with one
wavefront setting in the environment; every context says, when it is freed, that its
last call ran on that engine (the wavefront engine scans rows, the merging engine
does not)."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1311_0378_gb300 as rc  # noqa: E402
import test_gpu_fullsize as fullsize  # noqa: E402
import test_gpu_host_pipeline as pipeline  # noqa: E402
import test_gpu_ops as ops  # noqa: E402
import test_gpu_parity as parity  # noqa: E402


@pytest.fixture(autouse=True)
def wavefront(monkeypatch):
    import paper_1311_0378_gb300.build as b
    b.build()
    monkeypatch.setenv("RECON_REVISIT_SCANS", "1")
    freed, free = [], rc.recon_free

    def checked_free(c):
        freed.append(rc.recon_get_work(c, 1)[0]["scan_rows"] > 0)
        return free(c)
    monkeypatch.setattr(rc, "recon_free", checked_free)
    yield
    assert freed and all(freed)


@pytest.mark.parametrize("name", ["batch64", "uneven1000"])
def test_full_batches(name):
    """RECON_FLAG_LEARNED plans inside recon_batch here, and the plain schedule does not."""
    fullsize.test_fullsize_batch_every_tile_matches_oracle(name)


@pytest.mark.parametrize("test", [pipeline.test_host_batch_in_segments_matches_oracle,
                                  pipeline.test_host_batch_reports_failing_tile_of_a_later_segment,
                                  pipeline.test_host_batch_learned_schedule_matches_oracle,
                                  pipeline.test_host_batch_failing_first_segment_then_normal_call,
                                  ops.test_host_entry_point_fill_holes, parity.test_back_to_back_batches_without_sync])
def test_host_pipeline_and_replay(test):
    test()


@pytest.mark.parametrize("learned", [False, True])
def test_mixed_batch(learned):
    ops.test_mixed_batch(learned)
