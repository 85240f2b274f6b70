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


# Tokens in clusters and a small eps: rows of the plan that differ from one another, so that a row taken for another, or a k-block left
# out, shows.  Kept tokens around multiples of 64 (tiles of own rows) and 128, in batches that leave SMs idle and in larger ones, where a CTA
# has many units one after another, with a ring of four tiles of own rows and (1100 tokens) of two; widths whose last unit has no
# columns in its second half.  Reference: the recursion in 64 bits
# on the tokens that were kept.
@pytest.mark.parametrize("lengths", [[84, 85, 87, 170, 171, 172, 3, 1], [84, 85, 87, 170, 171, 172, 3, 1] * 30, [64] * 200,
                                     [255, 257, 340, 343], [400] * 40, [1100, 84] * 25])
@pytest.mark.parametrize("d", [64, 136, 264, 392, 1096, 1280])
def test_rows_of_the_plan(lengths, d):
    dev, r, alpha, eps = torch.device("cuda", 0), 0.25, 0.5, 0.1
    gen = torch.Generator(device=dev).manual_seed(d + len(lengths))
    total = sum(lengths)
    X = torch.randn(8, d, generator=gen, device=dev)[torch.randint(0, 8, (total,), generator=gen, device=dev)]
    X = (X + 0.3 * torch.randn(total, d, generator=gen, device=dev)) * torch.exp(0.5 * torch.randn(total, 1, generator=gen, device=dev))
    X = X.bfloat16()
    start = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int32)
    offs = torch.from_numpy(start).to(dev)
    plan = binding.Plan(d, X.dtype, len(lengths), total, max(lengths), device=dev)
    out = binding.Outputs.allocate(total, len(lengths), d, X.dtype, dev)
    plan.run(X, offs, binding.make_params(None, dynamic=0, r_fixed=r, alpha=alpha, eps=eps), out)
    assert plan.query_status() == 0
    plan.close()
    first = out.out_offsets.cpu().numpy()
    for n in sorted(set(lengths)):
        images = [i for i, m in enumerate(lengths) if m == n]
        M = int(first[images[0] + 1] - first[images[0]])
        B = n - M
        assert M == max(1, n - int(np.floor(r * n + 0.5)))
        x = torch.stack([X[start[i]:start[i + 1]] for i in images]).double()
        kept = torch.stack([out.kept_idx[first[i]:first[i] + M] for i in images]).long()
        pruned = torch.stack([out.merged_idx[start[i] - first[i]:start[i] - first[i] + B] for i in images]).long()
        Y = torch.stack([out.Y[first[i]:first[i] + M] for i in images]).double()
        own = torch.gather(x, 1, kept[:, :, None].expand(-1, -1, d))
        if B == 0:
            assert torch.equal(Y, own)
            continue
        away = torch.gather(x, 1, pruned[:, :, None].expand(-1, -1, d))
        K = torch.full((len(images), M + 1, B + 1), 0.2, dtype=torch.float64, device=dev)
        K[:, :M, :B] = torch.nn.functional.normalize(own, dim=2) @ torch.nn.functional.normalize(away, dim=2).transpose(1, 2)
        K = torch.exp((K - 1.0) / eps)
        V = torch.full((len(images), B + 1, 1), float(np.exp(1.0 / eps)), dtype=torch.float64, device=dev)
        a, b = torch.ones(M + 1, 1, dtype=torch.float64, device=dev), torch.ones(B + 1, 1, dtype=torch.float64, device=dev)
        a[M], b[B] = B, M
        for _ in range(100):
            U = a / (K @ V)
            V = b / (K.transpose(1, 2) @ U)
        P = (alpha * U * K * V.transpose(1, 2))[:, :M, :B]
        # bf16 rounds alpha P and the result by 2^-8 of them at most; the scores' fp32 sums of d terms, divided by eps, and the fp32
        # recursion move P by 1e-4 of itself at most
        bound = 2.0 ** -8 * own.abs() + (2.0 ** -7 + 1e-4) * (P @ away.abs())
        assert bool(((Y - (own + P @ away)).abs() <= bound).all()), n
        if M >= 60:                                            # (the bound tells rows apart: with the next row's plan most rows break it)
            wrong = ((Y - (own + P.roll(1, 1) @ away)).abs() > bound).any(2)
            assert float(wrong.double().mean()) > 0.5, n
