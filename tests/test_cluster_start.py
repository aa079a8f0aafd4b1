"""Shared memory of another CTA of the cluster may be touched only once that CTA runs.  Every kernel that reaches for it waits for a cluster
barrier first; checked on the source, since what happens otherwise is undefined."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_18063_b200", "csrc")


def _kernels():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = open(path).read()
        starts = [m.start() for m in re.finditer(r"^__global__", text, re.M)]
        for a, b in zip(starts, starts[1:] + [len(text)]):
            body = re.sub(r"//[^\n]*", "", text[a:b])
            if re.search(r"map_shared_rank|map_to_cta", body):
                yield os.path.basename(path) + ":" + re.search(r"(\w+)\s*\((?:const __grid_constant__ )?\w+ \w+[,)]", body).group(1), body


@pytest.mark.parametrize("name,body", list(_kernels()), ids=lambda v: v if len(v) < 80 else "")
def test_a_cluster_barrier_comes_before_the_first_remote_store(name, body):
    first = re.search(r"cluster_wait\(\)|cluster\.sync\(\)", body)
    stores = [m.start() for m in re.finditer(r"\bleader\[[^;]*\] = |\*cluster\.map_shared_rank|st_async_f32", body)]
    assert stores and first and first.start() < min(stores), name
