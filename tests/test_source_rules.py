"""Rules that the CUDA sources keep, checked on their text (no GPU needed)."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1904_02205_b200", "csrc")


def _sources():
    for name in sorted(os.listdir(CSRC)):
        with open(os.path.join(CSRC, name)) as f:
            yield name, re.sub(r"//[^\n]*", "", f.read())


def test_no_load_takes_the_read_only_path():
    """Kernels that start before their predecessor has ended may read what it writes only through ordinary loads:
    the compiler may move a read-only load above the wait."""
    for name, text in _sources():
        assert "__ldg(" not in text and "ld.global.nc" not in text, name
        hits = re.findall(r"const\s+\w+\s*\*\s*(?:const\s+)?__restrict__\s+\w+", text)
        assert not hits, "%s: %s" % (name, hits)
