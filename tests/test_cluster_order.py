"""A CTA of a cluster may store into another's shared memory only once that CTA is known to run: every kernel with such
stores meets the cluster (waits at a barrier of it) before its first one.  Read from the sources: a CTA that starts late is
nothing a test can bring about."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_00392_b200", "csrc")
MEETS = r"ptx::cluster_sync_all\(\)|ptx::cluster_wait_started\(\)"


# (file, function, the first store into another CTA, or the call that leads to it)
@pytest.mark.parametrize("name,function,store", [("scores_umma", "scores_umma_kernel", "st_cluster_v4"),
                                                 ("sinkhorn_reg", "sinkhorn_reg_kernel", "reg_sinkhorn<"),
                                                 ("sinkhorn_rows", "sinkhorn_rows_kernel", "sr_iterate<"),
                                                 ("sinkhorn_stream", "sinkhorn_stream_kernel", "st_solve<"),
                                                 ("sinkhorn_tall", "sinkhorn_tall_solve", "st_cluster_f32"),
                                                 ("fused", "stage2_fused_kernel", "fused_sinkhorn<")])
def test_kernel_meets_its_cluster_before_it_stores_into_it(name, function, store):
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name + ".cuh")).read())
    body = text[re.search(r"\b%s\(" % function, text).start():]
    assert store in body
    assert re.search(MEETS, body[:body.index(store)])
