"""rtprune_run_host with a fixed ratio takes a batch through in groups of images (copies in, kernels and copies out of
different groups overlap): what the device entry point gives, whatever the cuts: indices
exactly, values to rounding (the order of some sums depends on the number of images).  Marked gpu."""
import pytest
import torch

from paper_2605_00392_b200 import binding, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lengths,dtype,r", [([400] * 11, torch.bfloat16, 0.25), ([37, 1, 900, 900, 2, 1156, 400, 256, 400, 64], torch.bfloat16, 0.4),
                                             ([1, 3000, 1], torch.bfloat16, 0.3), ([256] * 20, torch.float32, 0.3),
                                             ([700] * 5, torch.bfloat16, 0.0)])
def test_groups_equal_the_device_entry_point(lengths, dtype, r):
    import parity
    w = synth.ragged(lengths, dtype=dtype, params=dict(r_fixed=r))
    plan = binding.Plan(w.d, w.X.dtype, w.batch, w.total_tokens, w.max_tokens)
    try:
        a = parity.run_gpu(w, plan=plan).out
        for _ in range(2):
            b = parity.run_gpu(w, plan=plan, host_path=True).out
            n = int(a.out_offsets[w.batch])
            nb = w.total_tokens - n
            assert torch.equal(a.out_offsets, b.out_offsets) and torch.equal(a.counts, b.counts)
            assert torch.equal(a.kept_idx[:n], b.kept_idx[:n])
            ya, yb = a.Y[:n].float(), b.Y[:n].float()
            unit = 2.0 ** (-8 if dtype == torch.bfloat16 else -20)
            assert (ya - yb).abs().max() <= unit * yb.abs().max() and (dtype != torch.bfloat16 or (ya != yb).float().mean() < 1e-3)
            assert r > 0 or torch.equal(a.Y[:n], b.Y[:n])
            assert torch.equal(a.merged_idx[:nb], b.merged_idx[:nb])
            torch.testing.assert_close(a.stats[:, :5], b.stats[:, :5], rtol=1e-5, atol=1e-6)
            torch.testing.assert_close(a.merge_weight[:nb], b.merge_weight[:nb], rtol=1e-5, atol=0)
    finally:
        plan.close()


def test_an_error_between_the_groups_leaves_nothing_in_flight():
    """A group that fails after others have been enqueued: the error is returned, and once the caller's stream has been
    waited for no copy is on its way any more (the last group before the failure copies 15 MB out)."""
    w = synth.ragged([400] * 8, params=dict(r_fixed=0.25))
    X, batch, kept = w.X.repeat(20, 1).pin_memory(), 160, 300
    offsets = (torch.arange(batch + 1) * 400).to(torch.int32).pin_memory()
    plan = binding.Plan(w.d, X.dtype, batch, X.shape[0], 400)
    try:
        out = binding.Outputs.allocate(X.shape[0], batch, w.d, X.dtype, "cpu", pin=True)
        params = binding.make_params(None, dynamic=0, r_fixed=0.25)
        rows = 4 * (batch // 8) * kept                       # of the four groups ahead of the failure
        for _ in range(3):
            out.Y.fill_(77.0)
            plan.fail_group(4)
            with pytest.raises(binding.RtpruneError):
                plan.run_host(X, offsets, None, params, out)
            torch.cuda.current_stream().synchronize()
            last = out.Y[rows - 1].clone()
            torch.cuda.synchronize()
            assert torch.equal(out.Y[rows - 1], last) and not (last == 77.0).any()
            assert (out.Y[rows:] == 77.0).all()              # the failed group and those after it
        plan.fail_group(-1)
        plan.run_host(X, offsets, None, params, out)         # the plan stays usable
        torch.cuda.current_stream().synchronize()
        assert int(out.out_offsets[batch]) == batch * kept and not (out.Y[:batch * kept] == 77.0).any()
    finally:
        plan.close()
