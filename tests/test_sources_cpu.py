"""Rules of the device code that no run can be relied on to show."""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_no_kernel_reads_through_the_non_coherent_path():
    """Kernels are launched with programmatic stream serialisation: they are resident while the launch ahead writes what
    they are about to read, which the non-coherent path (__ldg, ld.global.nc, or a kernel's const __restrict__ parameter) does
    not allow, whatever is waited for.  A stale window length or cutoff would show once in many runs, if ever."""
    seen = 0
    for path in sorted(glob.glob(os.path.join(ROOT, "paper_2512_11280_b200", "csrc", "*.cu*"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        assert "__ldg" not in text and "ld.global.nc" not in text, path
        for kernel in re.split(r"__global__", text)[1:]:
            body = kernel[: kernel.find("\n}\n")]
            if "pdl_wait" in body or "griddepcontrol.wait" in body:
                seen += 1
                assert "__restrict__" not in kernel[: kernel.find("{")], path
    assert seen >= 10
