"""Rules that the kernels' sources keep (CPU only)."""
import pathlib
import re

import paper_2607_20507_gb300 as package

CSRC = pathlib.Path(package.__file__).parent / "csrc"


def test_no_load_assumes_unchanging_memory():
    """The kernels start while the one before them still writes their inputs, so none reads by ld.global.nc."""
    sources = [f for f in CSRC.iterdir() if f.suffix in (".cu", ".cuh")]
    assert len(sources) > 5
    for f in sources:
        assert not re.search(r"__ldg\s*\(|ld\.global\.nc|__restrict__", f.read_text()), f.name
