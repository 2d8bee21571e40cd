"""Rules that every kernel source keeps and that no result on one GPU can show."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2205_02491_gb300", "csrc")
SOURCES = {os.path.basename(p): re.sub(r"//[^\n]*", "", open(p).read())
           for p in sorted(glob.glob(os.path.join(CSRC, "*.cu*")) + glob.glob(os.path.join(CSRC, "*.h")))}


def test_no_copy_is_multicast():
    """Each CTA fetches its own tiles: the library also runs as one replica per rank on several GPUs."""
    for name, text in SOURCES.items():
        joined = re.sub(r'"\s*"', "", text)  # adjacent string literals
        for asm in re.findall(r"cp\.async\.bulk[^;]*", joined):
            assert "multicast" not in asm, name
