"""Every buffer-check site that pcz_device.cuh lists for debug builds is one that
some kernel checks."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2308_11759_gb300", "csrc")


def test_listed_sites_are_checked():
    text = {f: open(f).read() for f in glob.glob(os.path.join(CSRC, "*.cu*"))}
    comment = re.search(r"// skips|Sites:(.*?)\n// -{10}", text[os.path.join(CSRC, "pcz_device.cuh")], re.S).group(1)
    listed = {int(n) for n in re.findall(r"\b(\d) the ", comment)}
    assert listed
    code = "\n".join(re.sub(r"//[^\n]*|#define[^\n]*", "", t) for t in text.values())
    checked = {int(n) for n in re.findall(r"PCZ_CHECK\([^;{]*?, (\d)\)", code)}
    assert listed == checked
