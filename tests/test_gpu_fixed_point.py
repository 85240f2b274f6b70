"""The exit at the fixed point (an iteration that moves no dual by more than rounding ends the loop, Appendix C's
T = 100 being an upper limit) against the same kernel's own T = 100 iterations, for every Sinkhorn kernel at a
tile of the largest kind it takes.  The profiling record names the kernel that ran.  Marked gpu."""
import numpy as np
import pytest
import torch

from paper_2605_00392_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def parity():
    import parity as _p
    return _p


@pytest.fixture(scope="module")
def binding():
    from paper_2605_00392_b200 import binding as _b
    return _b


def _run(binding, plan, w, dev, **over):
    p = dict(w.params)
    p.update(over)
    fields = {k: (int(v) if k in ("dynamic", "iters", "form", "stop_at_fixed_point", "criterion", "schedule") else float(v))
              for k, v in p.items()}
    params = binding.make_params(torch.from_numpy(w.rho.copy()).to(dev), **fields)
    out = binding.Outputs.allocate(w.total_tokens, w.batch, w.d, w.X.dtype, dev)
    plan.run(w.X.to(dev), torch.from_numpy(w.offsets.copy()).to(dev), params, out)
    names = [n for n, _ in plan.profile_read()]
    assert plan.query_status() == 0
    return out, names


# (case, image lengths, dtype, d, fixed r, extra parameters, kernel that must run, weight rtol)
CASES = [
    # register-resident K, clusters of two: 200 x 200, the largest tile of a 400-token image
    ("reg", [400] * 6, torch.bfloat16, 1280, 0.5, {}, "sinkhorn_reg", 2e-6),
    # more images than clusters of the register kernel fit at once: rows over warps, a CTA per image
    ("rows", [400] * 80, torch.bfloat16, 1280, 0.25, {}, "sinkhorn_rows", 2e-6),
    # the same batch at the ratio cap: 200 x 200 tiles no longer fit one CTA's shared memory, two CTAs per image
    ("rows_at_cap", [400] * 80, torch.bfloat16, 1280, 0.5, {}, "sinkhorn_rows", 2e-6),
    # 578 columns (more than 255): the instance for wide tiles, eight CTAs per image
    ("rows_wide", [1156, 1156, 900], torch.bfloat16, 1280, 0.5, {}, "sinkhorn_rows_wide", 2e-6),
    # 1729 columns: warps stream rows of K from the workspace (exit within 4 units: long sums)
    ("stream", [4512], torch.bfloat16, 1280, 0.3832, {}, "sinkhorn_stream", 2e-5),
    # 2256 columns, beyond that kernel: clusters of 8 or 16 CTAs iterate on K in the workspace (exit within 4 units)
    ("tall", [4512], torch.bfloat16, 1280, 0.5, {}, "sinkhorn_tall", 2e-5),
    # log-domain form, one CTA per image (exit when the duals repeat bit for bit)
    ("log", [400, 256], torch.bfloat16, 1280, 0.5, dict(form=1), "sinkhorn", 2e-5),
    # fp32 storage: rows over warps, the plan written in place
    ("fp32", [400] * 4, torch.float32, 64, 0.5, {}, "sinkhorn_rows", 2e-6),
]


@pytest.mark.parametrize("case", CASES, ids=[c[0] for c in CASES])
def test_exit_at_fixed_point_equals_all_iterations(binding, case):
    name, lengths, dtype, d, r, extra, kernel, wtol = case
    dev = torch.device("cuda", 0)
    w = synth.ragged(lengths, d=d, dtype=dtype, params=dict(r_fixed=r))
    plan = binding.Plan(w.d, w.X.dtype, w.batch, w.total_tokens, w.max_tokens, device=dev)
    plan.profile_enable(True)
    try:
        a, names_a = _run(binding, plan, w, dev, stop_at_fixed_point=1, **extra)
        b, names_b = _run(binding, plan, w, dev, stop_at_fixed_point=0, **extra)
    finally:
        plan.profile_enable(False)
        plan.close()
    assert kernel in names_a and names_a == names_b, (names_a, names_b)
    nb = w.batch
    ita, itb = a.stats[:nb, 5].cpu().numpy(), b.stats[:nb, 5].cpu().numpy()
    assert np.all(itb == 100.0), itb
    assert np.all(ita >= 1) and ita.max() < 100.0, ita          # the exit was taken
    assert torch.equal(a.kept_idx, b.kept_idx) and torch.equal(a.merged_idx, b.merged_idx)
    n = int(a.out_offsets[nb])
    npr = w.total_tokens - n
    wa, wb = a.merge_weight[:npr].cpu(), b.merge_weight[:npr].cpu()
    torch.testing.assert_close(wa, wb, rtol=wtol, atol=0)
    # partners: identical wherever the two runs' weights are not a rounding tie
    pa, pb = a.merge_partner[:npr].cpu(), b.merge_partner[:npr].cpu()
    differ = pa != pb
    assert float(differ.float().mean()) < 0.02, float(differ.float().mean())
    ya, yb = a.Y[:n].float().cpu(), b.Y[:n].float().cpu()
    if dtype == torch.bfloat16:
        assert (ya - yb).abs().max() <= 2.0 ** -8 * yb.abs().max()          # at most one bf16 rounding apart
        assert float((ya != yb).float().mean()) < 2e-3
    else:
        torch.testing.assert_close(ya, yb, rtol=1e-5, atol=1e-6)


# Where the iterations are many (eps below 1) the exit saves most and is reached slowly.  Once every dual settles, or all V but
# for a common factor, which leaves the plan as it is, an iteration moves V and with it U by 2^-23 of its value at most (against
# that factor), by four times that on images with more than 639 pruned tokens (the recursion does not expand a
# move), so what the 100 - k iterations that were saved can change in a weight is 2 (100 - k) such moves and the noise of its own
# factors.
@pytest.mark.parametrize("lengths,dtype,d,r,kernel", [([400] * 6, torch.bfloat16, 1280, 0.3, "sinkhorn_reg"),
                                                      ([256, 300] * 40, torch.bfloat16, 1280, 0.2, "sinkhorn_rows"),
                                                      ([1156, 456, 900], torch.bfloat16, 1280, 0.35, "sinkhorn_rows_wide"),
                                                      ([400, 256] * 4, torch.float32, 64, 0.25, "sinkhorn_rows"),
                                                      ([2137], torch.bfloat16, 1280, 0.4207, "sinkhorn_stream"),
                                                      ([4512], torch.bfloat16, 1280, 0.5, "sinkhorn_tall")])
@pytest.mark.parametrize("eps", [1.0, 0.3, 0.1, 0.05])
def test_exit_at_small_eps(binding, lengths, dtype, d, r, kernel, eps):
    dev = torch.device("cuda", 0)
    w = synth.ragged(lengths, d=d, dtype=dtype, params=dict(r_fixed=r))
    plan = binding.Plan(w.d, w.X.dtype, w.batch, w.total_tokens, w.max_tokens, device=dev)
    plan.profile_enable(True)
    try:
        a, names = _run(binding, plan, w, dev, stop_at_fixed_point=1, eps=eps)
        b, _ = _run(binding, plan, w, dev, stop_at_fixed_point=0, eps=eps)
    finally:
        plan.profile_enable(False)
        plan.close()
    assert kernel in names, names
    nb = w.batch
    k = a.stats[:nb, 5].cpu().numpy()
    assert np.all(b.stats[:nb, 5].cpu().numpy() == 100.0) and k.min() >= 1.0
    move, units = a.stats[:nb, 6].cpu().numpy(), 2.0 ** -23
    step = 4 if float(a.stats[:nb, 4].max()) > 639 else 1
    # (the reported move includes the common factor, which only rounding makes: the two sides' masses are equal)
    assert np.all(move[k < 100] <= 4 * units) and (eps < 0.3 or np.all(k < 100)), (k, move)
    offs, kept = w.offsets.astype(np.int64), a.out_offsets.cpu().numpy().astype(np.int64)
    wa, wb = a.merge_weight.cpu().numpy().astype(np.float64), b.merge_weight.cpu().numpy().astype(np.float64)
    for i in range(nb):
        s = slice(int(offs[i] - kept[i]), int(offs[i + 1] - kept[i + 1]))
        assert np.all(np.abs(wa[s] - wb[s]) <= (2 * step * (100 - k[i]) + 16) * units * wb[s]), (i, k[i], np.max(np.abs(wa[s] / wb[s] - 1)) / units)


# A token that is not a number (reported by the status word): its image leaves the loop when its duals, all NaN, repeat, and
# reports no move; the other images are what they are without it.
@pytest.mark.parametrize("batch,kernel", [(4, "sinkhorn_reg"), (160, "sinkhorn_rows_half")])
def test_an_image_that_is_not_a_number(binding, batch, kernel):
    dev = torch.device("cuda", 0)
    w = synth.ragged([100] * batch, d=1280, params=dict(r_fixed=0.25))
    plan = binding.Plan(w.d, w.X.dtype, w.batch, w.total_tokens, w.max_tokens, device=dev)
    X, offs = w.X.to(dev), torch.from_numpy(w.offsets.copy()).to(dev)
    params = binding.make_params(None, r_fixed=0.25)
    outs = [binding.Outputs.allocate(w.total_tokens, w.batch, w.d, w.X.dtype, dev) for _ in range(2)]
    plan.profile_enable(True)
    plan.run(X, offs, params, outs[0])
    assert plan.query_status() == 0 and kernel in [n for n, _ in plan.profile_read()]
    X[int(outs[0].merged_idx[3]), 5] = float("nan")            # a pruned token of the first image
    plan.run(X, offs, params, outs[1])
    assert plan.query_status() == binding.DEV_NONFINITE
    plan.profile_enable(False)
    plan.close()
    a, b = outs
    assert torch.isnan(b.stats[0, 0]) and b.stats[0, 5:7].tolist() == [2.0, 0.0]
    assert torch.equal(a.stats[1:], b.stats[1:]) and torch.equal(a.kept_idx[75:], b.kept_idx[75:])
    assert torch.equal(a.Y[75:75 * batch], b.Y[75:75 * batch]) and torch.equal(a.merge_weight[25:25 * batch], b.merge_weight[25:25 * batch])
