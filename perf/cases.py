"""The calls whose speed this framework answers for: twelve listed ones, and more of the same ranges on request.

  listed()            the listed cases, each a dict of plain values with a name
  draw(rng)           one more case of the same ranges
  prepare(case, seed) what a caller has in hand before the call: inputs and weights on the GPU (on the host for the host
                      entry point), the configuration, and the workspace it keeps
  run(state)          one call through the public entry points, and its outputs
  work(case)          bytes and flops that the call cannot do without
  tolerance(case)     how far two correct implementations may be apart

A case is (op, U users, up to C candidates each, L item rows per user, width d, H heads, segments of S items, M GSTA
layers, dtype).  d_qh = 16 per head everywhere.
"""
import math

import numpy as np
import torch

import paper_2602_11562_b200 as P

D_QH = 16
FFN_RATIO = 4       # hidden width of the feed-forward refinement, in units of d
NUM_RECENT = 2      # recent segment vectors in the fused output


def _case(name, op, U, C, L, d, H, S, M, dtype="bf16", lens="uniform", lo=0.25, ragged=False, dup=False):
    """lens: "full", "uniform" in [lo L, L], or "lognormal" (median 0.3 L, sigma 1, clipped to [L / 100, L]).
    ragged: candidate counts spread over [1, C] instead of C for every user.  dup: a tenth of the valid items are
    near-duplicates of one of the user's candidates and the gate is sharp enough to single them out."""
    c = dict(op=op, U=U, C=C, L=L, d=d, H=H, S=S, M=M, dtype=dtype, lens=lens, lo=lo, ragged=ragged, dup=dup)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: one user, a handful of candidates, fp32 (a check against another system, a debugging run);
        # latency and launches are all there is
        _case("tiny_f32", "forward", 1, 16, 256, 32, 1, 32, 1, dtype="f32", lens="full"),
        # a small fp32 batch of odd sizes
        _case("batch_f32", "forward", 5, 61, 777, 64, 4, 50, 2, dtype="f32", ragged=True),
        # online serving: one request, one user, a page of candidates
        _case("request", "forward", 1, 512, 2048, 64, 4, 64, 2, lo=0.5),
        # several requests of unequal size gathered into one call, items stored back to back, nothing a multiple of a tile
        _case("requests_packed", "packed", 29, 301, 1237, 96, 3, 37, 2, ragged=True),
        # batched ranking
        _case("ranking", "forward", 64, 256, 4096, 128, 4, 128, 2, lo=0.125, dup=True),
        # life-long histories, few users, many candidates
        _case("lifelong", "forward", 16, 1024, 10000, 64, 4, 100, 2, lens="lognormal"),
        # one candidate per user: scoring logged impressions
        _case("impressions", "forward", 4096, 1, 2048, 64, 2, 64, 1, lo=0.125),
        # the model's production shape (short segments), the whole compression stack: segment attention, feed-forward
        # refinement of the segment vectors, stacked attention, and the fused outputs the ranking tower reads
        _case("production_stack", "stack", 64, 256, 1000, 128, 2, 10, 2, lo=0.2),
        # batched ranking with the data in pinned host memory: what a process without GPU code of its own calls
        _case("ranking_host", "host", 64, 256, 4096, 128, 4, 128, 2, lo=0.125, dup=True),
        # training on batched ranking lists
        _case("train_lists", "backward", 64, 256, 4096, 128, 4, 128, 2, lo=0.125),
        # training on logged impressions: 2048 (user, target) pairs per GPU at the production shape
        _case("train_impressions", "backward", 2048, 1, 1000, 128, 2, 10, 2, lo=0.2),
        # a small fp32 training batch of odd sizes (gradient checks, fine-tuning of a small model)
        _case("train_f32", "backward", 6, 45, 600, 64, 2, 25, 2, dtype="f32", ragged=True),
    ]


_OPS = (["forward"] * 5 + ["packed"] * 2 + ["stack"] * 2 + ["host"] + ["backward"] * 3 + ["forward_f32"] * 2 + ["backward_f32"])


def draw(rng):
    """One more case: widths and head counts of the configurations in use, sizes log-uniform, cost at most that of the
    largest listed cases."""
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    while True:
        op = rng.choice(_OPS)
        dtype = "bf16"
        if op.endswith("_f32"):
            op, dtype = op[:-4], "f32"
        d = rng.choice([32, 64, 64, 96, 128, 128])
        H = d // rng.choice([w for w in (16, 32, 64) if d % w == 0 and d // w <= 8])
        L, S, M = log_int(64, 10000), log_int(5, 160), rng.choice([1, 2, 2, 3])
        if rng.random() < 0.2:
            U, C = log_int(16, 4096), 1
        else:
            U, C = log_int(1, 128), log_int(4, 1024)
        Lp = -(-L // S)
        if Lp > 128:
            continue
        rows, cands = U * L, U * C
        small = 32 if dtype == "f32" else 1
        elements = {"host": 6e7, "backward": 1.5e8}.get(op, 2.7e8)
        if rows * d > elements / small or cands * L * H > 4.5e8 / small or cands * Lp * d > 2.2e8 / small:
            continue
        if dtype == "f32" and Lp * d > 40000:        # (a candidate's segment vectors stay within one SM's shared memory)
            continue
        lens = rng.choice(["uniform", "uniform", "full", "lognormal"])
        return _case(None, op, U, C, L, d, H, S, M, dtype=dtype, lens=lens, lo=rng.choice([0.0, 0.1, 0.25, 0.5]),
                     ragged=C > 1 and rng.random() < 0.5)


def _torch_dtype(case):
    return torch.float32 if case["dtype"] == "f32" else torch.bfloat16


def _counts(case):
    """Candidates per user: a fixed multiset for a case (prepare() deals it out to the users)."""
    U, C = case["U"], case["C"]
    return np.random.default_rng(1000003 * U + C).integers(1, C + 1, size=U) if case["ragged"] else np.full(U, C)


def _lengths(case, rng):
    U, L = case["U"], case["L"]
    if case["lens"] == "full":
        n = np.full(U, L)
    elif case["lens"] == "uniform":
        n = rng.integers(int(case["lo"] * L), L + 1, size=U)
    else:
        n = np.clip(np.rint(np.exp(math.log(0.3 * L) + rng.standard_normal(U))), max(1, L // 100), L)
    return n.astype(np.int32)


def prepare(case, seed):
    U, C, L, d, H, M = (case[k] for k in ("U", "C", "L", "d", "H", "M"))
    dt, dev = _torch_dtype(case), torch.device("cuda")
    rng = np.random.default_rng(int(seed))
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(seed))
    lengths = _lengths(case, rng)
    counts = rng.permutation(_counts(case))
    offsets = np.concatenate([[0], np.cumsum(counts)]).astype(np.int32)
    N = int(offsets[-1])
    std = 1.0 / math.sqrt(d)

    items = torch.randn((U, L, d), generator=gen, device=dev, dtype=dt).mul_(std)
    cands = torch.randn((N, d), generator=gen, device=dev, dtype=dt).mul_(std)
    lengths_d = torch.from_numpy(lengths).to(dev)
    offsets_d = torch.from_numpy(offsets).to(dev)
    if case["dup"]:
        pick = (torch.rand((U, L), generator=gen, device=dev) < 0.1).nonzero()
        first, n = offsets_d[pick[:, 0]].long(), (offsets_d[pick[:, 0] + 1] - offsets_d[pick[:, 0]]).float()
        source = first + (torch.rand(len(pick), generator=gen, device=dev) * n).long().clamp_(max=C - 1)
        noise = torch.randn((len(pick), d), generator=gen, device=dev, dtype=dt).mul_(0.3 * std)
        items[pick[:, 0], pick[:, 1]] = cands[source] + noise
    valid = torch.arange(L, device=dev)[None, :] < lengths_d[:, None]
    if case["op"] != "packed":
        items.masked_fill_(~valid[:, :, None], 7.0)              # padding holds whatever the caller's buffer held

    def weights(*shape):
        a = math.sqrt(6.0 / (shape[-2] + shape[-1]))             # Xavier-uniform
        return torch.empty(shape, device=dev).uniform_(-a, a, generator=gen).to(dt)

    Wq, Wk, Wv, Wg = weights(d, H * D_QH), weights(d, H * D_QH), weights(d, d), weights(M, 3, d, d)
    if case["dup"]:
        Wk = Wq.clone()
    cfg = P.make_config(num_users=U, max_len=L, d_model=d, d_qk=H * D_QH, num_heads=H, seg_size=case["S"],
                        num_gsta_layers=M, dtype=case["dtype"], total_cands=N, max_cands_per_user=int(counts.max()),
                        sta_gamma=1.0 / 48.0 if case["dup"] else 0.0)
    s = {"op": case["op"], "cfg": cfg}

    def workspace(n):
        return torch.empty(n, dtype=torch.uint8, device=dev)

    if case["op"] == "host":
        s["args"] = tuple(t.cpu().pin_memory() for t in (items, lengths_d, cands, offsets_d, Wq, Wk, Wv, Wg))
        s["z"] = torch.empty((N, d), dtype=dt).pin_memory()
        s["workspace"] = workspace(P.laser_host_workspace_bytes(cfg))
        return s
    s["args"] = (items, lengths_d, cands, offsets_d, Wq, Wk, Wv, Wg)
    if case["op"] == "packed":
        starts = torch.from_numpy(np.concatenate([[0], np.cumsum(lengths)]).astype(np.int32)).to(dev)
        s["args"] = (items[valid].contiguous(), starts) + s["args"][1:]
    if case["op"] == "stack":
        hid = FFN_RATIO * d

        def vector(n, mean, spread):
            return (torch.randn(n, generator=gen, device=dev) * spread + mean).to(dt)

        s["ffn"] = {"W1": weights(d, hid), "b1": vector(hid, 0.0, 0.05), "W2": weights(hid, d), "b2": vector(d, 0.0, 0.05),
                    "ln_g": vector(d, 1.0, 0.1), "ln_b": vector(d, 0.0, 0.1)}
        s["workspace"] = workspace(P.laser_ffn_workspace_bytes(cfg, hid))
        s["fusion_workspace"] = workspace(256)
    elif case["op"] == "backward":
        s["dz"] = torch.randn((N, d), generator=gen, device=dev)
        s["workspace"] = workspace(P.laser_backward_workspace_bytes(cfg))
    else:
        s["workspace"] = workspace(P.laser_workspace_bytes(cfg))
    return s


def run(s):
    op, cfg, args = s["op"], s["cfg"], s["args"]
    if op == "forward":
        return P.laser_forward(cfg, *args, workspace=s["workspace"])
    if op == "packed":
        return P.laser_forward_packed(cfg, *args, workspace=s["workspace"])
    if op == "host":
        return P.laser_forward_host(cfg, *args, s["z"], s["workspace"])
    if op == "backward":
        return P.laser_backward(cfg, *args, s["dz"], workspace=s["workspace"])
    Hp, z = P.laser_forward_ffn(cfg, *args, s["ffn"], workspace=s["workspace"], want_hprime=True)
    fused = P.laser_fusion_forward(cfg, Hp, z, args[1], args[3], NUM_RECENT, workspace=s["fusion_workspace"])
    return {"Hprime": Hp, "fused": fused}


def _mean_length(case):
    if case["lens"] == "full":
        return float(case["L"])
    if case["lens"] == "uniform":
        return 0.5 * (int(case["lo"] * case["L"]) + case["L"])
    return 0.41 * case["L"]                                      # (median 0.3 L, sigma 1, clipped at L)


def work(case):
    U, L, d, H, S, M = (case[k] for k in ("U", "L", "d", "H", "S", "M"))
    es = 4 if case["dtype"] == "f32" else 2
    dqk, n = H * D_QH, _mean_length(case)
    N = int(_counts(case).sum())
    C, items, segs = N / U, U * n, n / S + 0.5
    # per item: keys and values once and a gate and a multiply-add per candidate, or (few candidates) both projections
    # folded into the query; per candidate and layer: three d x d products and two passes over its segment vectors
    flops = items * min(2 * d * (dqk + d) + 2 * (dqk + d) * C, 4 * H * d * C)
    flops += N * (2 * d * dqk + M * (6 * d * d + 4 * H * segs * d))
    weights = d * (2 * dqk + d + 3 * M * d)
    by = es * (items * d + N * d + weights) + 4 * (2 * U + 1)
    if case["op"] == "backward":
        return {"bytes": by + 4 * (U * L * d + 2 * N * d + weights), "flops": 3 * flops}
    if case["op"] == "stack":
        flops += N * segs * 4 * d * FFN_RATIO * d
        by += es * (N * -(-L // S) * d + N * (2 + NUM_RECENT) * d + 2 * FFN_RATIO * d * d)
        return {"bytes": by, "flops": flops}
    return {"bytes": by + es * N * d, "flops": flops}


def tolerance(case):
    if case["dtype"] == "f32":
        return {"rel": 1e-5, "max": 2e-4}       # fp32 products and sums throughout
    if case["op"] == "backward" and _counts(case).max() < 8:
        return {"rel": 2e-3, "max": 0.05}       # bf16 inputs, products of fp32 intermediates with TF32 operands
    if case["op"] == "backward":
        return {"rel": 2e-2, "max": 0.4}        # a chain of products with bf16 operands in the gates and the attention
    return {"rel": 1e-2, "max": 0.1}            # bf16 operands, intermediates and results
