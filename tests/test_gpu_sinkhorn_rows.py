"""The Sinkhorn kernel that shares an image's rows out over warps, where its lane layouts change (31/32, 63/64, 127/128,
255/256, 383/384, 511/512, 639/640 pruned tokens), with few and many rows beside them, rows that leave shared memory, and
one to eight CTAs per image.  fp32 storage and a small width keep the oracle short.  Marked gpu."""
import pytest
import torch

from paper_2605_00392_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lengths,r,iters", [([62, 64, 66, 126, 128, 254, 256, 3, 2], 0.5, 100), ([510, 512, 514, 30], 0.5, 100),
                                             ([766, 768, 1022], 0.5, 60), ([1024, 1278, 1280], 0.5, 40),
                                             ([700, 64, 33], 0.04, 100), ([300, 150], 0.9, 100), ([1100] * 40, 0.25, 8)])
def test_layout_edges(lengths, r, iters):
    import parity
    w = synth.ragged(lengths, d=64, dtype=torch.float32, params=dict(r_fixed=r, iters=iters))
    parity.check_workload(w, images=list(range(min(len(lengths), 9))))


def test_hand_over_to_the_merge_with_mixed_cluster_sizes():
    import parity
    w = synth.ragged([1156, 40, 456, 1, 900, 300], params=dict(dynamic=1, phi_lo=0.0, phi_hi=0.5, r_max=0.5))
    w.rho[4] = 1.0                                 # nothing to prune
    parity.check_workload(w)


# More CTAs than SMs and tiles of up to 255 columns: CTAs of 256 threads, two to an SM, at the same edges of lane layouts, one per
# image or (600 images) two; tiles that half an SM does not hold go to the whole one.
@pytest.mark.parametrize("lengths,r,iters", [([62, 64, 66, 126, 128, 200, 3, 2] * 20, 0.5, 100), ([69] * 150, 0.5, 100),
                                             ([254, 256, 30] * 60, 0.4, 30), ([400] * 600, 0.25, 30), ([510] * 150, 0.5, 20)])
def test_half_size_ctas(lengths, r, iters):
    import parity
    w = synth.ragged(lengths, d=64, dtype=torch.float32, params=dict(r_fixed=r, iters=iters))
    parity.check_workload(w, images=list(range(8)) + [len(lengths) - 1])
