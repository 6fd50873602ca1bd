"""The bench's renderer arms: what is called the 3DGS baseline evaluates every list entry at every pixel, and rows say
whether they skip entries per pixel block."""
import bench


def test_the_fp32_baseline_walks_every_entry():
    rows = {label: (prec, early, cull) for label, prec, early, cull in bench.ABLATION}
    assert rows["fp32"] == ("fp32", False, False)
    assert bench.ARMS["fp32"] == ("fp32", {"tile_cull": False})
    assert bench.ARMS["fp32_block_marks"] == ("fp32", {"tile_cull": True})


def test_rows_report_their_block_marks():
    for label, prec, _, cull in bench.ABLATION:
        if "block_marks" in label or prec == "fp32":
            assert bench.has_block_marks(prec, cull) == ("block_marks" in label), label
    assert not bench.has_block_marks("tc_fp16_global", True)
