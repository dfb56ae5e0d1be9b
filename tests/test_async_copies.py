"""A kernel waits for all its asynchronous copies before it ends: a block's
shared memory is given to the next block when its threads are done.  Shown on
the source of every kernel that issues cp.async."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2212_10733_gb300", "csrc")


def kernels(text):
    """(name, body) of every __global__ function, without comments."""
    text = re.sub(r"//[^\n]*", "", text)
    text = re.sub(r"__(?:launch_bounds|cluster_dims)__\s*\([^)]*\)", "", text)
    for m in re.finditer(r"__global__\b[^;{]*?(\w+)\s*\([^;{]*\)\s*\{", text):
        depth, j = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(text[j], 0)
            j += 1
        yield m.group(1), text[m.end():j]


def test_every_kernel_with_asynchronous_copies_ends_with_a_wait_for_all():
    found = {}
    for f in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        for name, body in kernels(open(f).read()):
            if re.search(r"cp\.async\.c[ag]\.shared", body):
                found[name] = body
    assert "rice_unpack_kernel" in found
    for name, body in found.items():
        waits = [m.start() for m in re.finditer(r"cp\.async\.wait_all|cp\.async\.wait_group 0", body)]
        # after the last statement that may start a copy, outside every loop
        assert waits and body[waits[-1]:].count("{") == 0 and body[waits[-1]:].count("}") == 1, name
        assert re.search(r"\bask\s*\(|commit_group", body[waits[-1]:]) is None, name
