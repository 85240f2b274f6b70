"""The textual-density kernel where its 256 x 64 tiles end and where its fp32 comparison must give way to the exact
one.  Counts bit-exact against the oracle, as in test_gpu_density.py.  Marked gpu."""
import numpy as np
import pytest
import torch

from oracle import density as od
from paper_2605_00392_b200 import binding

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda", 0)


@pytest.mark.parametrize("batch,height,width,patch", [(1, 16, 16, 16), (2, 80, 272, 16), (1, 96, 288, 32), (3, 64, 576, 64),
                                                      (40, 144, 528, 16), (24, 192, 1344, 64), (80, 128, 256, 32)])
def test_tile_edges(batch, height, width, patch):
    rng = np.random.default_rng(height + width)
    pages = rng.integers(0, 256, size=(batch, height, width, 3), dtype=np.uint8)
    pages[:, ::3] //= 2                                    # gradients on both sides of the threshold
    rho, counts, per_patch = binding.density(torch.from_numpy(pages).to(DEV), patch, 1.3, want_patch_counts=True)
    _, ref = od.density_batch(pages, patch, float(np.float32(1.3)))
    np.testing.assert_array_equal(per_patch.cpu().numpy(), ref)
    np.testing.assert_array_equal(counts.cpu().numpy(), ref.sum(axis=(1, 2)))


def test_gradients_next_to_the_threshold():
    # a vertical step: every pixel beside it has the same integer gradient; thresholds a few fp32 steps around it
    page = np.full((1, 64, 64, 3), 200, dtype=np.uint8)
    page[:, :, 30:] = (90, 31, 7)
    gray = lambda c: 299 * c[0] + 587 * c[1] + 114 * c[2]
    g = 4 * (gray((200, 200, 200)) - gray((90, 31, 7)))
    tau0 = np.float32(g / 255000.0)
    for k in range(-4, 5):
        tau = tau0
        for _ in range(abs(k)):
            tau = np.nextafter(tau, np.float32(10.0 if k > 0 else 0.0), dtype=np.float32)
        _, counts, _ = binding.density(torch.from_numpy(page).to(DEV), 64, float(tau))
        assert int(counts[0]) == (128 if float(g) ** 2 >= np.ceil((float(tau) * 255000.0) ** 2) else 0), k


def test_a_wait_that_gives_up_marks_its_image():
    # every CTA of every image gives up at once: no count may pass for a result
    pages = torch.randint(0, 256, (3, 128, 320, 3), dtype=torch.uint8, device=DEV)
    for patch in (16, 64):
        rho = torch.zeros(3, device=DEV)
        counts = torch.zeros(3, dtype=torch.int32, device=DEV)
        per_patch = torch.zeros(3 * (128 // patch) * (320 // patch), dtype=torch.int32, device=DEV)
        assert binding.lib().rtprune_test_density_expired(None, pages.data_ptr(), 3, 128, 320, patch, 0.2, rho.data_ptr(),
                                                          counts.data_ptr(), per_patch.data_ptr()) == 0
        torch.cuda.synchronize()
        assert torch.isnan(rho).all() and (counts == -1).all()             # (UINT32_MAX)
        rho, counts, per_patch = binding.density(pages, patch, 0.2, want_patch_counts=True)
        _, ref = od.density_batch(pages.cpu().numpy(), patch, float(np.float32(0.2)))
        np.testing.assert_array_equal(per_patch.cpu().numpy(), ref)
        assert torch.isfinite(rho).all()
