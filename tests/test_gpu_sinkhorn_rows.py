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


# More images than SMs and tiles of up to 255 columns: CTAs of 256 threads, two to an SM, at the same edges of lane layouts, with K in
# shared memory or (400 tokens) partly in L2; in bf16 storage plans and the hand-over to the merge too, ragged and dynamic.  A CTA
# per SM again (no length has r N within 32 bits' rounding of a half, 0.35 x 30 = 10.5 would):
# more than three eighths in L2, or any in a batch of little more than a wave, tiles of more than one CTA, more than 255 columns, and large
# tiles of a small batch at a small eps.
RAGGED = [62, 64, 66, 126, 128, 200, 3, 2]


@pytest.mark.parametrize("lengths,d,dtype,params,kernel", [
    (RAGGED * 20, 64, torch.float32, dict(r_fixed=0.5), "sinkhorn_rows_half"),
    ([69] * 150, 64, torch.float32, dict(r_fixed=0.5), "sinkhorn_rows_half"),
    ([254, 256, 30] * 60, 64, torch.float32, dict(r_fixed=0.4, iters=30), "sinkhorn_rows_half"),
    ([400] * 600, 64, torch.float32, dict(r_fixed=0.25, iters=30), "sinkhorn_rows_half"),
    (RAGGED * 20, 1280, torch.bfloat16, dict(r_fixed=0.5), "sinkhorn_rows_half"),
    ([400, 31, 280, 1, 333] * 52, 1280, torch.bfloat16, dict(r_fixed=0.35), "sinkhorn_rows_half"),
    ([256, 99, 180] * 51, 1280, torch.bfloat16, dict(dynamic=1, phi_lo=0.0, phi_hi=0.5, r_max=0.5), "sinkhorn_rows_half"),
    (RAGGED * 20, 1280, torch.bfloat16, dict(r_fixed=0.25, eps=0.1), "sinkhorn_rows_half"),
    (RAGGED * 20, 1280, torch.bfloat16, dict(r_fixed=0.5, eps=0.1), "sinkhorn_rows"),
    ([400] * 150, 1280, torch.bfloat16, dict(r_fixed=0.25, iters=20), "sinkhorn_rows"),
    ([400] * 260, 1280, torch.bfloat16, dict(r_fixed=0.5, iters=20), "sinkhorn_rows"),
    ([508] * 150, 64, torch.float32, dict(r_fixed=0.5, iters=20), "sinkhorn_rows"),
    ([510] * 150, 64, torch.float32, dict(r_fixed=0.5, iters=20), "sinkhorn_rows_wide")])
def test_half_size_ctas(lengths, d, dtype, params, kernel):
    import parity
    from paper_2605_00392_b200 import binding
    w = synth.ragged(lengths, d=d, dtype=dtype, params=params)
    plan = binding.Plan(w.d, w.X.dtype, w.batch, w.total_tokens, w.max_tokens)
    try:
        plan.profile_enable(True)
        parity.check_workload(w, plan=plan, images=list(range(8)) + [len(lengths) - 1])
        names = [n for n, _ in plan.profile_read()]
        assert [n for n in names if n.startswith("sinkhorn")] == [kernel], names
        plan.profile_enable(False)
    finally:
        plan.close()
