"""Every wait of a kernel is bounded: what the sources may hold, checked as text."""
import glob
import os
import re

from paper_1810_09958_gb300 import build


def kernel_sources():
    for path in sorted(glob.glob(os.path.join(build.CSRC, "*.cu*"))):
        with open(path) as f:
            yield os.path.basename(path), re.sub(r"//[^\n]*", "", f.read())


def test_no_barrier_joins_warps_that_may_have_given_up():
    """A warp whose bounded wait ran out leaves its loop, so a plain named
    barrier could hold the warps that wait for it for ever."""
    for name, text in kernel_sources():
        assert "bar.sync" not in text and "barrier.sync" not in text, name


def test_only_the_depthwise_loop_keeps_a_named_barrier():
    """Its warps come to it whatever their waits said, and leave together.  In the
    GEMM's split epilogue a warp could leave at the accumulator's wait while the
    others went on to the barrier."""
    users = [name for name, text in kernel_sources() if re.search(r"\bnamed_bar_and\(", text) and name != "ptx.cuh"]
    assert users == ["depthwise.cu"], users


def test_every_wait_for_a_tensor_memory_load_names_its_registers():
    """The load fills its registers asynchronously: work on them could otherwise
    be moved ahead of the wait."""
    for name, text in kernel_sources():
        assert "tmem_ld_wait()" not in text, name
        for asm in re.findall(r'"tcgen05\.wait::ld[^;]*;"\s*:(.)', text):
            assert asm != ":", name


def test_error_sites_belong_to_one_kernel_each():
    """isam_sync reports the site and block alone."""
    sites = [(code, name) for name, text in kernel_sources()
             for code in re.findall(r"\bSITE_\w+ = (0x[0-9A-Fa-f]+)", text) + re.findall(r"\b(0x[0-9A-Fa-f]{3})u\)", text)]
    codes = [int(code, 16) for code, _ in sites]
    assert len(codes) > 40 and len(set(codes)) == len(codes), sorted(sites)
