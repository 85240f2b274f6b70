"""The Sinkhorn kernel that streams score tiles of 640 to 2047 pruned tokens, where its widths change (a multiple of 256
columns with the dustbin's), with few rows (warps and CTAs without any) and many, clusters of 2 to 16 CTAs.  fp32 storage
and a small width keep the oracle short.  Marked gpu."""
import pytest
import torch

from paper_2605_00392_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lengths,r,iters", [([1278, 1280, 1282], 0.5, 12), ([1534, 1536], 0.5, 12), ([2048, 2046], 0.5, 8),
                                             ([2100, 2600, 3070], 0.4999, 6), ([4094], 0.5, 5), ([700, 641, 642], 0.9985, 30),
                                             ([2000], 0.99, 10), ([1300] * 40, 0.5, 6), ([1300] * 80, 0.5, 3), ([1500, 20], 0.5, 0),
                                             ([1500], 0.5, 1)])
def test_edges(lengths, r, iters):
    import parity
    w = synth.ragged(lengths, d=64, dtype=torch.float32, params=dict(r_fixed=r, iters=iters))
    parity.check_workload(w, images=list(range(min(len(lengths), 3))))


def test_all_iterations_and_tolerance():
    import parity
    w = synth.ragged([1600], d=64, dtype=torch.float32, params=dict(r_fixed=0.45))
    a = parity.run_gpu(w, overrides=dict(stop_at_fixed_point=0)).out
    b = parity.run_gpu(w, overrides=dict(tol=1e-3)).out
    assert float(a.stats[0, 5]) == 100.0 and 1.0 <= float(b.stats[0, 5]) <= 5.0 and float(b.stats[0, 6]) <= 1e-3


@pytest.mark.parametrize("lengths,d,dtype,r,iters", [([1400, 700, 30], 1280, torch.bfloat16, 0.5, 100), ([2137], 1280, torch.bfloat16, 0.4207, 100),
                                                     ([1400] * 20, 64, torch.float32, 0.5, 30), ([3000, 4094], 64, torch.float32, 0.5, 6)])
def test_without_a_cluster_of_the_kernel_the_one_for_wider_tiles_runs(lengths, d, dtype, r, iters):
    import parity
    from paper_2605_00392_b200 import binding
    w = synth.ragged(lengths, d=d, dtype=dtype, params=dict(r_fixed=r, iters=iters))
    plan = binding.Plan(w.d, w.X.dtype, w.batch, w.total_tokens, w.max_tokens)
    try:
        plan.no_stream_clusters()
        plan.profile_enable(True)
        parity.check_workload(w, plan=plan, images=list(range(min(len(lengths), 3))))
        names = [n for n, _ in plan.profile_read()]
        assert "sinkhorn_tall" in names and "sinkhorn_stream" not in names
        plan.profile_enable(False)
    finally:
        plan.close()


# Scores from the copy of the kept rows (more than 639 pruned tokens possible, room for d columns in a plan row of max_tokens
# rounded up to 64): kept rows around a whole number of 128-row tiles, pruned ones around whole passes of 256 columns, an image
# that another kernel solves and some with next to nothing to prune beside them; the last has no room for the copy.
@pytest.mark.parametrize("lengths,r,d", [([1536, 1538, 1300, 1, 40], 0.5, 1280), ([1408, 1406], 0.5, 1408), ([1400, 60], 0.5, 1416)])
def test_scores_of_kept_rows(lengths, r, d):
    import parity
    w = synth.ragged(lengths, d=d, dtype=torch.bfloat16, params=dict(r_fixed=r, iters=10))
    parity.check_workload(w)
