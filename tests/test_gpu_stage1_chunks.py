"""Stage 1 where the tokens per CTA follow the batch: images of different lengths (by their mean: clamped to 32 and to 512
tokens, and between), a little more than a wave of equal ones, equal ones through a plan made for longer images.  Norms, counts and phi against torch in 64 bits.  Marked gpu."""
import numpy as np
import pytest
import torch

from paper_2605_00392_b200 import binding

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lengths,most", [([456, 1156, 33, 700] * 16, 1156), ([1, 40, 97], 97), ([1100, 300] * 200, 1100), ([64] * 310, 64),
                                          ([65] * 370, 65), ([65] * 371, 65), ([257] * 444, 257), ([257] * 445, 257), ([400] * 64, 4512), ([100], 1156), ([69] * 300, 400)])
def test_norms_counts_and_phi(lengths, most):
    d, dev = 64, torch.device("cuda", 0)
    total, batch = sum(lengths), len(lengths)
    gen = torch.Generator(device=dev).manual_seed(total)
    X = torch.randn(total, d, generator=gen, device=dev) + 0.5
    offs = torch.from_numpy(np.concatenate([[0], np.cumsum(lengths)]).astype(np.int32)).to(dev)
    plan = binding.Plan(d, torch.float32, batch, total, most, device=dev)
    out = binding.Outputs.allocate(total, batch, d, torch.float32, dev)
    params = binding.make_params(torch.full((batch,), 0.6, device=dev), dynamic=1, r_fixed=0.0, phi_lo=0.0, phi_hi=1.0, r_max=0.5)
    plan.run(X, offs, params, out)
    assert plan.query_status() == 0
    plan.close()
    kept = out.out_offsets.cpu().numpy()
    for i, x in enumerate(torch.split(X.double(), list(lengths))):
        n, norm = len(x), x.norm(dim=1)
        s = (x / norm[:, None]).sum(0)
        phi = float((s @ s - n) / max(n * (n - 1), 1))
        # a sum of n unit vectors in 32 bits: n d roundings of 2^-24 at the most, in practice far fewer
        assert abs(float(out.stats[i, 0]) - phi) <= 2e-6 * max(1.0, abs(phi)), (i, n)
        m = int(out.counts[i])
        assert kept[i + 1] - kept[i] == m and 1 <= m <= n
        want = torch.sort(torch.argsort(norm.float(), descending=True, stable=True)[:m])[0]
        got = out.kept_idx[kept[i]:kept[i + 1]].long()
        assert float((norm[got].sum() - norm[want].sum()).abs()) <= 1e-5 * float(norm.sum())     # (near-ties may swap)
