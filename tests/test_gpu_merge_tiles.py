"""The merge of bf16 storage at the edges of its tiles: kept tokens around multiples of 128, widths around 128 and 256 columns,
nothing pruned, one k-block to many, against the merge of fp32 storage on the same values.  Marked gpu."""
import numpy as np
import pytest
import torch

from paper_2605_00392_b200 import binding

pytestmark = pytest.mark.gpu


def _run(X, offs, r, alpha, lengths):
    dev, d = X.device, X.shape[1]
    plan = binding.Plan(d, X.dtype, len(lengths), X.shape[0], max(lengths), device=dev)
    out = binding.Outputs.allocate(X.shape[0], len(lengths), d, X.dtype, dev)
    plan.run(X, offs, binding.make_params(None, dynamic=0, r_fixed=r, alpha=alpha), out)
    assert plan.query_status() == 0
    plan.close()
    n = int(out.out_offsets[-1])
    return out.kept_idx[:n], out.Y[:n]


@pytest.mark.parametrize("lengths,r", [([1, 2, 127, 128, 129, 255, 256, 257], 0.0), ([183, 184, 185, 366, 367, 64, 3, 1], 0.3),
                                       ([126, 128, 130, 254, 256, 258, 512, 514], 0.5), ([900, 700, 20], 0.45), ([400] * 40, 0.25)])
@pytest.mark.parametrize("d", [64, 136, 256, 264, 392])
def test_tiles(lengths, r, d):
    dev = torch.device("cuda", 0)
    X = torch.randn(sum(lengths), d, generator=torch.Generator(device=dev).manual_seed(d), device=dev).bfloat16()
    offs = torch.from_numpy(np.concatenate([[0], np.cumsum(lengths)]).astype(np.int32)).to(dev)
    kept, Y = _run(X, offs, r, 0.0, lengths)                   # alpha = 0: the kept rows, bit for bit
    m = torch.tensor([n - int(np.floor(np.float32(r) * n + 0.5)) for n in lengths], device=dev)
    m = torch.maximum(m, torch.ones_like(m))
    rows = torch.repeat_interleave(offs[:-1].long(), m) + kept.long()
    assert torch.equal(Y, X[rows])
    kept, Y = _run(X, offs, r, 1.0, lengths)
    kept32, Y32 = _run(X.float(), offs, r, 1.0, lengths)
    same = kept == kept32                                      # (norms that differ in the last bits may rank either way)
    assert float(same.float().mean()) > 0.99
    # a row of the plan sums to 1 at most: its rounding to bf16 is 2^-9 of the largest |x|, that of y 2^-9 of |y|; doubled for
    # the scores' own rounding
    bound = 2.0 ** -8 * (Y32.abs() + X.float().abs().max())
    assert bool(((Y.float() - Y32).abs() <= bound)[same].all())
