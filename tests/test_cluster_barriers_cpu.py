"""Blocks of a cluster touch one another's shared memory only once all of them are known to run: in the source of every kernel a cluster
barrier stands before the first such access."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2408_15766_b200", "csrc")
REMOTE = re.compile(r"\b(?:st_cluster|ld_cluster)_\w+\s*\(|\bmerge_lists\b")      # (merge_lists reads the lists of all blocks)
BARRIER = re.compile(r"\bcluster_(?:sync|wait)\s*\(")


def kernels():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cuh"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for part in text.split("__global__")[1:]:
            yield re.search(r"(\w+)\s*\((?:const\s|int|unsigned|float)", part).group(1), part


def test_a_cluster_barrier_comes_before_the_first_remote_access():
    seen = []
    for name, body in kernels():
        remote = REMOTE.search(body)
        if remote is None:
            continue
        seen.append(name)
        barrier = BARRIER.search(body)
        assert barrier is not None and barrier.start() < remote.start(), name
    assert set(seen) >= {"gemm_kernel", "normed_kernel", "row_split_kernel", "hca_bwd_fused_kernel", "hca_attention_pair_kernel"}, seen
