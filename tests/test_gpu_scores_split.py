"""The scores of small batches, whose contraction is shared out over clusters of 4 CTAs: pruned counts around the
units of 16 columns, widths whose k-blocks do not share out evenly (or are fewer than the CTAs), images that end within a
tile.  Marked gpu."""
import pytest
import torch

from paper_2605_00392_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lengths,d,r", [([64], 1280, 0.25), ([129, 1], 1280, 0.12), ([400, 34, 512], 1280, 0.5), ([200], 1024, 0.08),
                                         ([300] * 8, 1536, 0.11), ([256] * 30, 1280, 0.3), ([70, 33], 264, 0.5), ([400] * 12, 1288, 0.64)])
def test_split_tiles(lengths, d, r):
    import parity
    w = synth.ragged(lengths, d=d, params=dict(r_fixed=r))
    parity.check_workload(w, images=list(range(min(4, len(lengths)))))
