"""Kernels that may start before their predecessor on the stream has ended (launch_kernel with
`after`) wait for it before they read anything in global memory: an earlier kernel of the
same call may have written it, the schedule and the tables included. Read off the sources, on the CPU."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1504_05046_gb300", "csrc")


def _kernels():
    """(file, name, body) of every kernel whose body waits with grid_wait()."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__[^;{]*?\b(\w+)\s*\(const __grid_constant__ SplitArgs a[^)]*\)\s*\{", text):
            depth, end = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(text[end], 0)
                end += 1
            yield os.path.basename(path), m.group(1), text[m.end():end]


def test_nothing_is_read_before_the_wait():
    seen = set()
    for name, kernel, body in _kernels():
        assert body.count("grid_wait();") == 1, (name, kernel)
        before = body[:body.index("grid_wait();")]
        # an array of the arguments, indexed, dereferenced or handed to a load
        reads = re.findall(r"\ba\.\w+\s*\[|\*\s*a\.\w+|__ldg\(|\ba\.prods\b", before)
        assert not reads, (name, kernel, reads)
        seen.add(kernel)
    assert {"split_exp_kernel", "split_exp_lines_kernel", "split_scale_lines_kernel", "split_pack_kernel",
            "split_mma_kernel", "split_mma_wide_kernel", "split_reduce_kernel"} <= seen
