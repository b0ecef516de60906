"""Loads of the CUDA sources, read as text.  A kernel launched as a programmatic
dependent (``pdl_wait``) is alive while the step before it writes the set that it
reads, so no population and no status word may be read by a non-coherent load
(``__ldg``, ``ld.global.nc``), nor by a plain read through a pointer to const
__restrict__, which the compiler may turn into one.  The __half forms of the
header's cached loads are not volatile and may move across the wait."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2208_03562_gb300", "csrc")


def sources():
    for p in sorted(glob.glob(os.path.join(CSRC, "*.cu*")) + glob.glob(os.path.join(CSRC, "*.h"))):
        with open(p) as f:
            yield os.path.basename(p), re.sub(r"//[^\n]*", "", f.read())


def test_no_non_coherent_loads():
    for name, text in sources():
        assert not re.search(r"__ldg\s*\(|ld\.global\.nc", text), name


def test_cached_loads_of_halves_are_volatile():
    for name, text in sources():
        assert not re.search(r"__ldc[ag]\s*\((?=[^;]*half)", text), name
    text = dict(sources())["prc_device.cuh"]
    loads = re.findall(r"asm( volatile)?\s*\(\"ld\.global[^\"]*\"", text)
    assert len(loads) == 10 and all(loads)


def test_status_flag_is_read_by_a_coherent_load():
    for name, text in sources():
        for kernel in text.split("__global__")[1:]:
            if "pdl_wait()" in kernel and "const DevStatus *" in kernel.split("{")[0]:
                assert not re.search(r"(?<!&)\bst->stop", kernel), name
