"""A block of a thread-block cluster may write into another block's shared
memory only after a cluster barrier has shown that the other one has started.
Shown on the source: in every kernel with cluster dimensions the first
statement that can reach a remote store comes after a barrier.  (A store to a
block that has not started is undefined, so nothing here runs it.)"""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2212_10733_gb300", "csrc")
REMOTE = re.compile(r"\b(?:put_u64|put_u32|cluster_sums|process_cluster)\s*\(|shared::cluster")


def bodies(text):
    """(name, body) of every kernel with __cluster_dims__, without comments."""
    text = re.sub(r"//[^\n]*", "", text)
    for m in re.finditer(r"__cluster_dims__\s*\(", text):
        name = re.compile(r"(\w+)\s*\(\s*const\s").search(text, m.end())
        i = text.index("{", name.end())
        depth, j = 1, i + 1
        while depth:
            depth += {"{": 1, "}": -1}.get(text[j], 0)
            j += 1
        yield name.group(1), text[i:j]


def test_a_cluster_barrier_precedes_the_first_remote_store():
    found = [b for f in sorted(glob.glob(os.path.join(CSRC, "*.cu")))
             for b in bodies(open(f).read())]
    assert "fused_fp64_cluster_kernel" in [n for n, _ in found]
    for name, body in found:
        use = REMOTE.search(body)
        barrier = body.find("cluster_sync()")
        assert use is None or 0 <= barrier < use.start(), name
