"""The work that users of the library have it do, as cases that can be prepared, run and compared.

A case is a dict of plain values.  `kind` says which public entry point it goes through:

  run      Plan.run on device buffers (bf16 or fp32 storage)
  host     Plan.run_host: pinned host buffers in, pinned host buffers out, and the wait for them
  density  binding.density: the textual density of page images, the input rho of the dynamic ratio

Inputs have the structure the method meets on document pages: text tokens of many directions and large
norms, background tokens that are near-duplicates of one another with small norms.  Neighbouring sorted
norms are at least 1.5e-3 apart and rho puts r N on an integer, so that which tokens are kept does not
hang on the last bit of a sum; the background tokens differ enough (cosines 0.99 with a spread of 3e-4)
that the partner of a pruned token rarely does.
"""
import math

import numpy as np
import torch

from paper_2605_00392_b200 import binding

GOLDEN = 0.6180339887498949
CLUSTERS = 16                 # text directions per page
NORM_GAP = 1.5e-3
PHI_HI, R_MAX = 0.737, 0.5    # the dynamic ratio as the repository's own configurations set it
STATS_USED = 5                # phi, rho, r, M, B; the other columns say how the iteration went, not what came out


def _run(name, batch, n_lo, n_hi, step, dynamic, ratio, dtype="bf16", d=1280, eps=1.0, kind="run"):
    return {"name": name, "kind": kind, "batch": batch, "n_lo": n_lo, "n_hi": n_hi, "step": step, "dynamic": dynamic,
            "ratio": ratio, "dtype": dtype, "d": d, "eps": eps}


def listed():
    return [
        # the smallest request a user makes: one thumbnail of 64 tokens on its way into a prefill that waits for it
        _run("thumbnail 1x64", 1, 64, 64, 1, False, 0.25),
        # the ordinary interactive request: one page at the large resolution mode, dynamic ratio
        _run("page 1x400", 1, 400, 400, 1, True, 0.0),
        # a serving engine's batch at the base resolution mode
        _run("batch 32x256", 32, 256, 256, 1, True, 0.0),
        # the same at the large resolution mode: the headline batch of the repository's benchmark
        _run("batch 64x400", 64, 400, 400, 1, True, 0.0),
        # multi-view pages: 256 global tokens + 2 to 9 tiles of 100, lengths mixed within the batch
        _run("multi-view 128x456-1156", 128, 456, 1156, 100, True, 0.0),
        # offline processing of a corpus in the largest batches, fixed retention 0.75
        _run("corpus 1024x400", 1024, 400, 400, 1, False, 0.25),
        # fp32 storage: encoders whose features must not be rounded
        _run("fp32 256x400", 256, 400, 400, 1, True, 0.0, dtype="fp32"),
        # models with large visual token sets: 2137 tokens of which 1238 are kept, 4512 of which 2783 are kept
        _run("long 16x2137", 16, 2137, 2137, 1, False, 0.4207),
        _run("long 8x4512", 8, 4512, 4512, 1, False, 0.3832),
        # a sharper transport plan (eps 0.1): many more iterations per page
        _run("sharp 64x456-1156", 64, 456, 1156, 100, True, 0.0, eps=0.1),
        # features that live on the host: copies in, the path at the fixed retention, copies out, the wait
        _run("host 64x400", 64, 400, 400, 1, False, 0.25, kind="host"),
        # the step before: textual density, per patch and per page, of the pages of one large batch
        {"name": "density 64x1280x1280", "kind": "density", "batch": 64, "height": 1280, "width": 1280, "patch": 64},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    family = rng.choice(["run"] * 6 + ["long"] * 2 + ["fp32", "sharp", "host", "density"])
    if family == "density":
        patch = rng.choice([16, 32, 64])
        return {"kind": "density", "batch": _log_int(rng, 1, 64), "height": patch * rng.randint(512 // patch, 1280 // patch),
                "width": patch * rng.randint(512 // patch, 1280 // patch), "patch": patch}
    d = rng.choice([1280, 1280, 1280, 1024, 1536])
    most_tokens = {"run": 1024 * 400 * 1280 // d, "long": 34000, "fp32": 256 * 400, "sharp": 50000, "host": 64 * 400}[family]
    if family == "long":
        n_hi, most_batch = _log_int(rng, 1200, 4512), 16
    elif family == "sharp":
        n_hi, most_batch = _log_int(rng, 256, 1156), 64
    elif family == "run":
        n_hi, most_batch = _log_int(rng, 64, 1156), 1024
    else:
        n_hi, most_batch = _log_int(rng, 64, 400), 256 if family == "fp32" else 64
    most_batch = min(most_batch, most_tokens // n_hi, 145_000_000 * 1280 // (n_hi * n_hi * d))
    batch = _log_int(rng, 1, max(1, most_batch))
    n_lo = n_hi if rng.random() < 0.5 else max(16, int(n_hi * rng.uniform(0.3, 0.9)))
    dynamic = family not in ("long", "host") and rng.random() < 0.6
    c = _run("", batch, n_lo, n_hi, 1, dynamic, 0.0 if dynamic else round(rng.uniform(0.1, 0.5), 4),
             dtype="fp32" if family == "fp32" else "bf16", d=d, eps=0.1 if family == "sharp" else 1.0,
             kind="host" if family == "host" else "run")
    del c["name"]
    return c


def lengths(case):
    """Tokens of each image: spread evenly over [n_lo, n_hi] in steps of `step`, in mixed order."""
    steps = (case["n_hi"] - case["n_lo"]) // case["step"] + 1
    return [case["n_lo"] + case["step"] * int(((i + 1) * GOLDEN % 1.0) * steps) for i in range(case["batch"])]


def _tokens(case, seed):
    """X [sum N, d] on the GPU, offsets, rho: see the head of the file."""
    dev = torch.device("cuda", torch.cuda.current_device())
    gen = torch.Generator(device=dev).manual_seed(seed)
    lens, d, batch = lengths(case), case["d"], case["batch"]
    total = sum(lens)
    offsets = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    n_of = torch.tensor(lens, device=dev)
    img = torch.repeat_interleave(torch.arange(batch, device=dev), n_of, output_size=total)
    density = 0.2 + 0.7 * torch.rand(batch, generator=gen, device=dev)              # share of text tokens per image
    text = torch.rand(total, generator=gen, device=dev) < density[img]
    centres = torch.randn(batch * (CLUSTERS + 1), d, generator=gen, device=dev)       # the last of each: background
    which = torch.randint(0, CLUSTERS, (total,), generator=gen, device=dev)
    which = torch.where(text, which, torch.full_like(which, CLUSTERS)) + img * (CLUSTERS + 1)
    # norms: log-normal, background half as large; then neighbours in an image's sorted order moved apart
    logn = 0.5 * torch.randn(total, generator=gen, device=dev) + 0.5 * math.log(d)
    logn = (logn - math.log(2.0) * (~text)).double()
    key, order = torch.sort(logn + 1000.0 * img)
    start = torch.tensor(offsets[:-1].astype(np.int64), device=dev)
    rank = torch.arange(total, device=dev) - start[img]          # place within the image (the sort is image-major)
    apart = torch.cummax(key - NORM_GAP * rank, dim=0)[0] + NORM_GAP * rank - 1000.0 * img
    norm = torch.empty(total, dtype=torch.float64, device=dev)
    norm[order] = torch.exp(apart)
    norm = norm.float()
    dtype = torch.float32 if case["dtype"] == "fp32" else torch.bfloat16
    X = torch.empty(total, d, dtype=dtype, device=dev)
    for a in range(0, total, 1 << 17):
        b = min(total, a + (1 << 17))
        rows = torch.randn(b - a, d, generator=gen, device=dev)
        rows.mul_(torch.where(text[a:b], 0.5, 0.1)[:, None]).add_(centres[which[a:b]])
        X[a:b] = rows.mul_((norm[a:b] / rows.norm(dim=1))[:, None]).to(dtype)
    # rho: the page's text density, moved to where r N is a whole number
    rho = torch.zeros(batch, dtype=torch.float32)
    if case["dynamic"]:
        sums = torch.stack([torch.nn.functional.normalize(x.double(), dim=1).sum(0) for x in torch.split(X, lens)])
        n = np.array(lens, dtype=np.float64)
        phi = ((sums * sums).sum(1).cpu().numpy() - n) / np.maximum(n * (n - 1.0), 1.0)
        f = np.clip(phi / PHI_HI, 1e-6, 1.0)
        pruned = np.floor(np.minimum(f * (1.0 - density.double().cpu().numpy()), R_MAX) * n)
        rho = torch.from_numpy(1.0 - pruned / n / f).float()
    return X, torch.from_numpy(offsets), rho


def _pages(case, seed):
    """Near-white pages with faint noise and, in some 64 x 64 patches, lines of dark sharp-edged dots."""
    dev = torch.device("cuda", torch.cuda.current_device())
    gen = torch.Generator(device=dev).manual_seed(seed)
    b, h, w = case["batch"], case["height"], case["width"]

    def rand(*shape):
        return torch.rand(*shape, generator=gen, device=dev)

    def grow(mask, y, x):
        return mask.repeat_interleave(y, 1).repeat_interleave(x, 2)[:, :h, :w]

    share = 0.2 + 0.7 * rand(b, 1, 1)
    ink = grow(rand(b, -(-h // 64), -(-w // 64)) < share, 64, 64) & grow(rand(b, -(-h // 16), -(-w // 8)) < 0.55, 16, 8)
    line = torch.arange(h, device=dev) % 16
    ink &= ((line >= 3) & (line <= 12))[None, :, None]
    ink &= rand(b, h, w) < 0.34
    noise = torch.randint(-2, 2, (b, h, w), generator=gen, device=dev)
    pages = torch.empty(b, h, w, 3, dtype=torch.uint8, device=dev)
    for ch in range(3):
        paper = torch.randint(240, 252, (b, 1, 1), generator=gen, device=dev)
        black = torch.randint(10, 80, (b, 1, 1), generator=gen, device=dev)
        pages[..., ch] = (torch.where(ink, black, paper) + noise).to(torch.uint8)
    return pages


def prepare(case, seed):
    if case["kind"] == "density":
        return {"kind": "density", "pages": _pages(case, seed), "patch": case["patch"]}
    X, offsets, rho = _tokens(case, seed)
    dev, total, batch, d = X.device, X.shape[0], case["batch"], case["d"]
    plan = binding.Plan(d, X.dtype, batch, total, max(lengths(case)), device=dev)
    ratio = dict(dynamic=1, r_fixed=0.0, phi_lo=0.0, phi_hi=PHI_HI, r_max=R_MAX) if case["dynamic"] \
        else dict(dynamic=0, r_fixed=case["ratio"])
    if case["kind"] == "host":
        out = binding.Outputs.allocate(total, batch, d, X.dtype, "cpu", pin=True)
        return {"kind": "host", "plan": plan, "X": X.cpu().pin_memory(), "offsets": offsets.pin_memory(),
                "rho": rho.pin_memory(), "params": binding.make_params(None, eps=case["eps"], **ratio), "out": out}
    rho = rho.to(dev)
    out = binding.Outputs.allocate(total, batch, d, X.dtype, dev)
    out.Y.zero_()                  # rows past the kept ones are never written
    return {"kind": "run", "plan": plan, "X": X, "offsets": offsets.to(dev), "rho": rho,
            "params": binding.make_params(rho if case["dynamic"] else None, eps=case["eps"], **ratio), "out": out}


def run(state):
    if state["kind"] == "density":
        rho, counts, patch_counts = binding.density(state["pages"], state["patch"], 0.2, want_patch_counts=True)
        return {"rho": rho, "counts": counts, "patch_counts": patch_counts}
    plan, out = state["plan"], state["out"]
    if state["kind"] == "host":
        plan.run_host(state["X"], state["offsets"], state["rho"], state["params"], out)
        torch.cuda.current_stream().synchronize()            # host outputs may be read from here on
        kept = int(out.out_offsets[-1])                        # rows past these are not meaningful
        pruned = out.Y.shape[0] - kept
        return {"Y": out.Y[:kept], "out_offsets": out.out_offsets, "counts": out.counts, "kept_idx": out.kept_idx[:kept],
                "merged_idx": out.merged_idx[:pruned], "merge_partner": out.merge_partner[:pruned],
                "merge_weight": out.merge_weight[:pruned], "stats": out.stats[:, :STATS_USED]}
    plan.run(state["X"], state["offsets"], state["params"], out)
    return {"Y": out.Y, "out_offsets": out.out_offsets, "counts": out.counts, "kept_idx": out.kept_idx,
            "merged_idx": out.merged_idx, "merge_partner": out.merge_partner, "merge_weight": out.merge_weight,
            "stats": out.stats[:, :STATS_USED]}


def work(case):
    """Each input read once, each output written once; the two contractions of the second stage and five
    Sinkhorn iterations, the fewest such an image takes.  A dynamic ratio keeps about 0.84 of the tokens."""
    if case["kind"] == "density":
        pixels = case["batch"] * case["height"] * case["width"]
        return {"bytes": 3.0 * pixels + 8.0 * case["batch"], "flops": 20.0 * pixels}
    size = 4 if case["dtype"] == "fp32" else 2
    nbytes = flops = 0.0
    for n in lengths(case):
        pruned = 0.16 * n if case["dynamic"] else math.floor(case["ratio"] * n + 0.5)
        nbytes += (2 * n - pruned) * case["d"] * size + 12.0 * n + 44.0
        flops += 4.0 * (n - pruned) * pruned * case["d"] + 3.0 * n * case["d"] + 5 * 4.0 * (n - pruned) * pruned
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    if case["kind"] == "density":
        return "exact"
    if case["dtype"] == "fp32":
        return {"rel": 1e-5, "max": 1e-4, "differ": 0.01}
    # bf16 rows: half a unit in the last place is 2^-9 of a value; partners of near-tied columns may differ
    return {"rel": 4e-3, "max": 2e-2, "differ": 0.01}
