"""Compiler flags of single files: only the unit whose values have to match the device's bit for bit is compiled
without contraction; the FP64 transform behind every Fresnel axis is not in it."""
import os

from paper_1107_5578_gb300 import build


def test_contraction_is_off_in_the_asm_entries_alone():
    off = sorted(f for f, flags in build.FILE_FLAGS.items() if "-ffp-contract=off" in flags)
    assert len(off) == 1 and off[0] in build.CPP_SOURCES
    text = open(os.path.join(build.CSRC, off[0])).read()
    assert "asm_axis_entry" in text
    for other in ("fft64", "fresnel_axis_dft", "shifted_fresnel_axis"):
        assert other not in text
