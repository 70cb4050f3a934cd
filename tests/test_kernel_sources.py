"""What the kernels' sources promise by how they read memory (no GPU)."""

import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_34244_gb300", "csrc")


def test_dependent_kernels_read_only_the_tables_through_the_read_only_path():
    """A kernel launched behind another (launch_after) runs while that one
    still writes the worklist: griddepcontrol.wait orders ordinary loads, not
    the read-only path (__ldg), which needs data that nothing writes while the
    kernel runs.  Only the screen, launched the ordinary way, reads its inputs
    so; every other __ldg reads a table of the image (built before the call)."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        if os.path.basename(path) in ("heddle_price.cu", "heddle_noalloc.cu"):  # nothing here is launched behind
            assert "launch_after(" not in open(path).read()
            continue
        text = re.sub(r"//[^\n]*", "", open(path).read())
        tables = set(re.findall(r"\b(\w+) = reinterpret_cast<const \w+\*>\(\w+\.img \+", text))
        for arg in re.findall(r"__ldg\(([^()]*)\)", text):
            base = arg.split("+")[0].strip()
            assert base in tables, "%s: __ldg(%s)" % (os.path.basename(path), arg)


def test_every_search_checks_that_its_split_attains_the_bound():
    """A threshold search that returned a bound above B* would report it with a
    split that keeps it; each of the three raises the consistency flag unless
    the split's largest stage time equals the bound."""
    for name in ("heddle_eqsearch.cu", "heddle_gsearch.cu", "heddle_wsearch.cu"):
        text = open(os.path.join(CSRC, name)).read()
        assert re.search(r"tmax != Bstar\) atomicOr\(a\.err, kErrInternal\)", text), name
