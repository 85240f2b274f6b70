"""The top-M selection by counted ranks (images of up to 256 tokens) at its edges, ties included, against a stable sort.
Marked gpu."""
import numpy as np
import pytest
import torch

from paper_2605_00392_b200 import binding

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("criterion", [0, 2])
@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 64, 255, 256, 257, 288, 400, 511, 512, 513])
def test_kept_tokens_in_index_order(n, criterion):
    dev = torch.device("cuda", 0)
    rng = np.random.default_rng(n)
    X = rng.standard_normal((3 * n, 64)).astype(np.float32)
    X[n:2 * n] = X[n:n + max(1, n // 7)][rng.integers(0, max(1, n // 7), n)]       # many equal tokens
    X[2 * n:] = X[2 * n]                                                            # all equal
    plan = binding.Plan(64, torch.float32, 3, max(3 * n, 24), max(n, 8))
    out = binding.Outputs.allocate(3 * n, 3, 64, torch.float32, dev)
    c = torch.zeros(3 * n, device=dev)
    order = torch.zeros(3 * n, dtype=torch.int32, device=dev)
    offs = torch.tensor([0, n, 2 * n, 3 * n], dtype=torch.int32, device=dev)
    for r in (0.0, 0.3, 0.999):
        plan.select(torch.from_numpy(X).to(dev), offs, binding.make_params(r_fixed=r, criterion=criterion), out, c, order)
        assert plan.query_status() == 0
        for i in range(3):
            key, got, M = c[i * n:(i + 1) * n].cpu().numpy(), order[i * n:(i + 1) * n].cpu().numpy(), int(out.counts[i])
            ranked = np.argsort(-key, kind="stable")
            np.testing.assert_array_equal(got, np.concatenate([np.sort(ranked[:M]), np.sort(ranked[M:])]))
    plan.close()
