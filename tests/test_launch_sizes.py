"""Grids of persistent kernels and rounds of blocks follow the device: with fewer SMs than a number in
the code the last blocks of a persistent kernel would start only after the first round."""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_no_source_assumes_a_number_of_sms():
    for path in glob.glob(os.path.join(ROOT, "paper_2509_07974_gb300", "csrc", "*.cu*")):
        code = re.sub(r"//[^\n]*|/\*.*?\*/", "", open(path).read(), flags=re.S)
        assert not re.search(r"\b152\b", code), os.path.basename(path)
