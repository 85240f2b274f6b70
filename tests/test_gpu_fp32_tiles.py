"""fp32 storage where the tiles of its tensor-core contractions end: kept rows around 128, pruned tokens around 64 and 128
(k-blocks of the merge, and where it stops holding the split plan in shared memory), widths that leave a part of a
64-column block, more output tiles than a task takes.  Marked gpu."""
import pytest
import torch

from paper_2605_00392_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lengths,d,r", [([128, 129, 127, 2, 1], 64, 0.004), ([192, 256, 257, 258], 132, 0.5), ([321, 130], 68, 0.4),
                                         ([64, 700], 4, 0.45), ([200, 90], 1284, 0.3)])
def test_tile_edges(lengths, d, r):
    import parity
    w = synth.ragged(lengths, d=d, dtype=torch.float32, params=dict(r_fixed=r))
    parity.check_workload(w)
