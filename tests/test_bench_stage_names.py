"""The bench names the search that ran: the filtered one whatever option led to
it, the split search only where its two passes ran."""
import bench


def test_stage_kernel():
    for tuned in (None, "split", "split_scan", "automatic", "grouped"):
        assert bench.stage_kernel(tuned, True) == "automatic"
    assert bench.stage_kernel("split", False) == bench.stage_kernel("split_scan", False) == "split"
    assert bench.stage_kernel("grouped", False) == "grouped"
    assert bench.stage_kernel("automatic", False) is None and bench.stage_kernel(None, False) is None
