"""Reads of tensor memory are warp-collective: whatever the lanes did before (a wait each spun on for itself, a
branch that some rows took), the warp has to be together, and with one outcome of the wait, when it issues one.
Checked on the sources: a violation is undefined behaviour, which a run need not show."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2110_00625_b200", "csrc")


def _functions(text):
    """(name, body) of the inline functions at the outermost level."""
    return re.findall(r"^__device__ __forceinline__ \w+ (\w+)\([^{]*\) \{\n(.*?)^\}", text, flags=re.S | re.M)


def test_every_read_brings_the_warp_together_first():
    functions = _functions(open(os.path.join(CSRC, "tc_ptx.cuh")).read())
    reads = [(n, b) for n, b in functions if "tcgen05.ld.sync" in b or "tcgen05.wait::ld" in b]
    assert {n for n, _ in reads} >= {"tmem_ld_32x32", "tmem_ld_16cols", "tmem_ld_8cols", "tmem_ld_wait"}
    for name, body in reads:
        assert "__syncwarp();" in body.split("asm volatile")[0], name


def test_reads_are_issued_through_those_functions():
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        if not path.endswith("tc_ptx.cuh"):
            text = open(path).read()
            assert "tcgen05.ld.sync" not in text and "tcgen05.wait::ld.sync" not in text, path


def test_a_warp_that_reads_after_a_wait_has_one_outcome_of_it():
    # the waits of the epilogue warps (their error codes say who waits); single lanes wait elsewhere
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        for line in open(path).read().splitlines():
            if not re.search(r"ERR_(WG_)?EPILOGUE[,)]", line) or "mbar_wait" not in line:
                continue
            alone = "failed = true" in line or "lane == 0" in line or "z_part" in line
            assert alone or "mbar_wait_warp" in line or "__all_sync" in line, (path, line)
