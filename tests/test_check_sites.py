"""The bounds-checked build names a failed check by its site code: one code per place."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1504_05022_gb300", "csrc")


def test_site_codes_are_unique():
    codes = []
    for f in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        codes += re.findall(r"SPG_IN\([^;]*?, (\d+)\)", open(f).read())
    assert len(codes) >= 18
    assert sorted(codes) == sorted(set(codes))
