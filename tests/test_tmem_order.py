"""Order of a tensor-core kernel's beginning, read from its source: tensor memory is the block's own (allocation, then a barrier of the whole
block) before the block lets the blocks of the next kernel in (nf_pdl_begin).  Those allocate theirs and hold it while they wait for
this grid to end, so a block that let them in first could wait for its columns without end."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2402_14139_b200", "csrc")


def _kernels():
    """(file, name, body) of every kernel of the library that allocates tensor memory."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for part in text.split("__global__")[1:]:
            if "tmem_alloc(" in part:
                yield os.path.basename(path), re.search(r"(\w+)\s*\(const __grid_constant__", part).group(1), part


def test_tensor_memory_is_allocated_before_dependents_may_start():
    found = list(_kernels())
    assert len(found) >= 8
    for path, name, body in found:
        begin = body.index("nf_pdl_begin()")
        alloc = body.rindex("tmem_alloc(", 0, begin)
        assert "__syncthreads()" in body[alloc:begin], (path, name)
        assert "launch_dependents" not in body[:begin], (path, name)
