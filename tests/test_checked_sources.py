"""The bounds-checked build sees every voxel load of the tracers: they go
through the device helpers that hold the check, kfetch and brick_fetch."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1902_01137_gb300", "csrc")


def test_tracers_load_voxels_through_the_checked_helpers():
    for name in ("trace.cu", "wavefront.cu"):
        text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
        raw = re.findall(r"[^\n]*\b[SZ]\.vox(?:16)?\b[^\n]*", text)     # (the scene's; F.vox are queue entries)
        assert not raw, (name, raw)


def test_leaf_entries_name_a_checked_brick():
    # a voxel leaf's brick comes from the leaf map: the checked build compares it with the voxel's own
    text = open(os.path.join(CSRC, "mcrt_device.cuh")).read()
    body = text[text.index("brick_fetch("):]
    checked = body[body.index("#ifdef MCRT_CHECKED"):body.index("#else")]
    assert "MCRT_CHECK" in checked and "brick ==" in checked
