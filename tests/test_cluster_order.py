"""Clusters and tensor memory, by reading the kernels' source.

A CTA that holds tensor-memory columns while it waits for its cluster can wait without end for a CTA
of another kernel's cluster that does the same (each holds what the other's peer is waiting for).  So
every kernel that allocates columns and meets its cluster gives them back first.
"""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1409_0940_gb300", "csrc")
ALLOC = re.compile(r"tmem_alloc<1>|tcgen05\.alloc\.cta_group::1")
RELEASE = re.compile(r"tmem_return(_and_meet)?\(|tmem_dealloc<1>|tcgen05\.dealloc\.cta_group::1")
# a wait for the cluster (tmem_return_and_meet waits after its release; CTA pairs hold their columns, and
# an SM's shared memory with them, to the end)
BARRIER = re.compile(r"(?<!if \(CG == 2\) )(cluster_sync_all|cluster_wait)\(")


def kernels():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = open(path).read()
        starts = [m.start() for m in re.finditer(r"__global__", text)] + [len(text)]
        for a, b in zip(starts, starts[1:]):
            yield os.path.basename(path), text[a:b]


def test_the_helper_releases_before_it_waits():
    text = open(os.path.join(CSRC, "simt.cuh")).read()
    body = text[text.index("void tmem_return_and_meet("):]
    body = body[:body.index("\n}\n")]
    assert body.index("tmem_dealloc<1>") < body.index("cluster_wait()") and "cluster_sync_all" not in body


def test_tensor_memory_is_given_back_before_a_cluster_is_waited_for():
    seen = []
    for path, body in kernels():
        barrier = BARRIER.search(body)
        if not ALLOC.search(body) or not barrier:
            continue
        name = re.search(r"\b(k_\w+)\(", body).group(1)
        seen.append(name)
        before = [m.start() for m in RELEASE.finditer(body) if m.start() < barrier.start()]
        after = [m.start() for m in RELEASE.finditer(body) if m.start() > barrier.start()]
        assert before and not after, (path, name)
    assert sorted(seen) == ["k_gemm_f32_nn", "k_gram_tile", "k_pass2_simt", "k_split_gemm"]
