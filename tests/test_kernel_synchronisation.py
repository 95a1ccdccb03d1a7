"""A CTA may touch another CTA's shared memory only once that one is known to have started.  Read off the sources: a kernel
that breaks this goes wrong on rare runs only, if at all."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2007_10412_b200", "csrc")


def _kernels():
    """(file, kernel, body without comments) of every kernel in the sources."""
    out = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__[^;{]*?\b(\w+_kernel)\s*\([^{;]*\{", text, flags=re.S):
            depth, i = 1, m.end()
            while depth > 0:
                depth += {"{": 1, "}": -1}.get(text[i], 0)
                i += 1
            out.append((os.path.basename(path), m.group(1), text[m.end():i]))
    return out


REMOTE = r"\bst_cluster_\w+\s*\(|\bmbar_arrive_remote\s*\("
STORING = [k for k in _kernels() if re.search(REMOTE, k[2])]


def test_kernels_that_write_to_peers_are_found():
    assert {"xent_small_kernel", "store_index_small_kernel", "tc_gemm_pair_kernel", "tc_sparse_pair_kernel"} <= {k[1] for k in STORING}


@pytest.mark.parametrize("file,kernel,body", STORING, ids=[k[1] for k in STORING])
def test_peers_have_started_before_the_first_write_to_them(file, kernel, body):
    first = re.search(REMOTE, body).start()
    assert re.search(r"\bcluster_barrier\s*\(\s*\)|\bcluster_started_wait\s*\(\s*\)", body[:first]), (file, kernel)
    # ... and nobody leaves while a peer may still write to it
    last = [m.start() for m in re.finditer(REMOTE, body)][-1]
    assert "cluster_barrier()" in body[last:], (file, kernel)
