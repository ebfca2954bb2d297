"""What a user of this library has it do, as cases that can be timed and compared.

A case is one attention layer of a video diffusion transformer on a (T, Hh, W) token grid, called
through the package's entry points the way a model calls them.  The kinds of layer:

  layer      block scores -> top-k selection -> block-sparse attention
  merged     token merge -> (the model's own projection of the merged tokens) -> scores -> selection ->
             attention on the merged sequence -> unmerge back to the full grid
  statistic  a layer that also writes the log-sum-exp and takes the key marginal and its entropy, which
             the sparsity scheduler reads
  branches   local-cube attention and long-range top-k attention computed apart and fused
  local      token merge with matching kept near the source's own block, the plan then applied to two
             more tensors of the layer through its cached lists, and one result unmerged

Inputs are a sum of eight travelling waves shared by all tensors of a case plus white noise, scaled by
d^-0.25, in bf16: neighbouring tokens are alike and queries and keys share structure, as in the
activations of a video model, so that selection and merging have something to find.
"""
import math

import torch

import paper_2512_05754_b200 as usv

BLOCK = usv.BLOCK


# ------------------------------------------------------------------------------------------ cases
def _case(kind, B, H, d, grid, keep, merge=0, part=(1, 1, 2), token_major=False, name=None):
    c = {"kind": kind, "B": B, "H": H, "d": d, "T": grid[0], "Hh": grid[1], "W": grid[2], "keep": keep,
         "merge": merge, "st": part[0], "sh": part[1], "sw": part[2], "token_major": token_major}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the sanity instance of the configurations: what a test or a first try runs; all latency
        _case("layer", 1, 2, 64, (4, 16, 16), "25", name="tiny_d64"),
        # a short low-resolution clip (2025 tokens, a partial last block), Q/K/V as views of one
        # projection output: latency and launches count
        _case("layer", 1, 12, 128, (5, 15, 27), "20", token_major=True, name="clip_2k"),
        # the headline layer: 480p, 32 760 tokens, keep 10 %
        _case("layer", 1, 12, 128, (21, 30, 52), "10", name="layer_480p"),
        # the same grid with half of the tokens merged first (alternate tokens as destinations)
        _case("merged", 1, 12, 128, (21, 30, 52), "10", merge=50, token_major=True, name="merged_480p"),
        # a 720p layer of a large model: many heads, 1182 key blocks a row
        _case("layer", 1, 40, 128, (21, 45, 80), "5", name="layer_720p"),
        # the largest: a 720p guidance pair, keep ratios from dense to 5 % on its heads, a quarter merged
        _case("merged", 2, 24, 128, (33, 45, 80), "100,25,10,5", merge=25, token_major=True, name="merged_720p_mixed"),
        # the longest sequence of the length sweep: 193 440 tokens, 3023 key blocks a row
        _case("layer", 1, 12, 128, (31, 60, 104), "5", name="layer_193k"),
        # head width 64, the other one the library takes, at the 480p grid with the same channels
        _case("layer", 1, 24, 64, (21, 30, 52), "10", name="layer_480p_d64"),
        # head width 64 with 2x2 spatial merging of a quarter of the tokens, odd grid (19 x 29 x 51)
        _case("merged", 1, 24, 64, (19, 29, 51), "15", merge=25, part=(1, 2, 2), token_major=True, name="merged_odd_d64"),
        # a calibration step of the scheduler at 480p: attention, then its entropy statistic
        _case("statistic", 1, 12, 128, (21, 30, 52), "10", name="statistic_480p"),
        # two-branch layer on a guidance pair of shorter clips
        _case("branches", 2, 12, 128, (13, 30, 52), "12", name="branches_clip"),
        # a plan made once and applied to several tensors: the bandwidth-bound side of merging
        _case("local", 2, 12, 128, (21, 30, 52), "10", merge=40, name="local_merge_480p"),
    ]


def _most_work():
    return work(next(c for c in listed() if c["name"] == "merged_720p_mixed"))


def draw(rng):
    most = _most_work()
    while True:
        kind = rng.choice(["layer", "layer", "layer", "merged", "merged", "statistic", "branches", "local"])
        longest = 120000 if kind in ("merged", "local") else 200000
        n = math.exp(rng.uniform(math.log(700), math.log(longest)))
        T = max(1, round(math.exp(rng.uniform(0.0, math.log(33)))))
        Hh = max(4, round(math.sqrt(n / T / rng.uniform(1.0, 2.0))))
        W = max(4, round(n / T / Hh))
        H = rng.choice([2, 3, 8, 12, 16, 24, 40])
        keep = rng.choice(["5", "10", "10", "20", "25", "35", "100,25,10,5", "100"])
        part = rng.choice([(1, 1, 2), (1, 2, 2), (2, 2, 2)])
        merge = 0
        if kind in ("merged", "local"):
            merge = rng.choice([10, 25, 40] + ([50] if part != (1, 1, 2) else []))
        c = _case(kind, rng.choice([1, 1, 2]), H, rng.choice([128, 128, 64]), (T, Hh, W), keep, merge, part,
                  token_major=(kind == "merged" or rng.random() < 0.3))
        w = work(c)
        if T * Hh * W >= 600 and w["bytes"] <= 0.5 * most["bytes"] and w["flops"] <= 0.15 * most["flops"]:
            return c


# ----------------------------------------------------------------------------------------- shapes
def _sizes(c):
    """(tokens, merged sources, tokens that attention sees, key blocks, kept key blocks per head)."""
    n = c["T"] * c["Hh"] * c["W"]
    r = c["merge"] * n // 100
    m = n - r if c["kind"] == "merged" else n
    nb = -(-m // BLOCK)
    ratios = [int(p) for p in c["keep"].split(",")]
    low = 2 if c["kind"] == "branches" and nb > 1 else 1
    k = [max(low, -(-ratios[h % len(ratios)] * nb // 100)) for h in range(c["H"])]
    return n, r, m, nb, k


def _destinations(c):
    return -(-c["T"] // c["st"]) * -(-c["Hh"] // c["sh"]) * -(-c["W"] // c["sw"])


# ----------------------------------------------------------------------------------------- inputs
def _field(gen, waves, grid, channels, d):
    """bf16 [T*Hh*W, channels]: sum over eight waves of a sin(w.p + phi), plus noise, times d^-0.25."""
    T, Hh, W = grid
    dev = gen.device
    t = torch.arange(T, device=dev, dtype=torch.float32)
    y = torch.arange(Hh, device=dev, dtype=torch.float32)
    x = torch.arange(W, device=dev, dtype=torch.float32)
    p = torch.cartesian_prod(t, y, x).reshape(-1, 3)
    phase = p @ waves.t()
    a = torch.randn((8, channels), generator=gen, device=dev)
    phi = 2 * math.pi * torch.rand((8, channels), generator=gen, device=dev)
    basis = torch.cat([phase.sin(), phase.cos()], 1)
    f = basis @ torch.cat([a * phi.cos(), a * phi.sin()], 0)
    f += 0.5 * torch.randn(f.shape, generator=gen, device=dev)
    return (f * float(d) ** -0.25).to(torch.bfloat16)


def _weight(gen, rows, cols):
    return (torch.randn((rows, cols), generator=gen, device=gen.device) / math.sqrt(rows)).to(torch.bfloat16)


def prepare(case, seed):
    c = case
    dev = torch.device("cuda", torch.cuda.current_device())
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    B, H, d, grid = c["B"], c["H"], c["d"], (c["T"], c["Hh"], c["W"])
    C = H * d
    n, r, m, nb, k = _sizes(c)
    waves = 0.5 * torch.rand((8, 3), generator=gen, device=dev)
    s = {"case": c, "k": k, "grid": grid, "part": (c["st"], c["sh"], c["sw"]), "r": r}
    if c["kind"] in ("merged", "local"):
        # hidden states and the layer's key projection, which is the metric tokens are matched by
        s["z"] = torch.stack([_field(gen, waves, grid, C, d) for _ in range(B)])
        wk = _weight(gen, C, C)
        s["metric"] = (s["z"] @ wk).reshape(B, n, H, d)
        if c["kind"] == "local":
            s["x2"] = s["z"] @ _weight(gen, C, C)
            s["x3"] = s["z"] @ _weight(gen, C, C)
            return s
        # Q, K, V of the merged tokens: what the model's projection hands to the attention
        zm, _ = usv.token_merge(s["z"], s["metric"], s["grid"], s["part"], r)
        w = torch.cat([_weight(gen, C, C), wk, _weight(gen, C, C)], 1)
        qkv = (zm @ w).reshape(B, m, 3, H, d)
        s["q"], s["k_"], s["v"] = (qkv[:, :, i].permute(0, 2, 1, 3) for i in range(3))
        return s
    for name in ("q", "k_", "v"):
        x = torch.stack([_field(gen, waves, grid, C, d) for _ in range(B)]).reshape(B, n, H, d).permute(0, 2, 1, 3)
        s[name] = x if c["token_major"] else x.contiguous()
    if c["kind"] == "branches":
        # the local branch's key-block list: every query block attends its own block
        s["own"] = torch.arange(nb, dtype=torch.int32, device=dev).view(1, 1, nb, 1).expand(B, H, nb, 1).contiguous()
        s["k_long"] = [x - 1 for x in k]
    return s


# ------------------------------------------------------------------------------------------- a pass
def run(state):
    s = state
    kind = s["case"]["kind"]
    if kind == "local":
        zm, plan = usv.token_merge(s["z"], s["metric"], s["grid"], s["part"], s["r"], window=(1, 1, 1))
        x2 = usv.token_merge_apply(s["x2"], plan)
        x3 = usv.token_merge_apply(s["x3"], plan)
        return {"z": zm, "x2": x2, "x3": x3, "y": usv.token_unmerge(x2, plan.pos), "dst_of": plan.dst_of, "pos": plan.pos}
    out = {}
    if kind == "merged":
        out["z"], plan = usv.token_merge(s["z"], s["metric"], s["grid"], s["part"], s["r"])
        out["dst_of"], out["pos"] = plan.dst_of, plan.pos
    q, k, v, kept = s["q"], s["k_"], s["v"], s["k"]
    scores = usv.block_scores(q, k)
    if kind == "branches":
        sel = usv.select_blocks(usv.exclude_own_block(scores), s["k_long"])
        o1, l1 = usv.sparse_attn_fwd(q, k, v, s["own"], [1] * len(kept), return_lse=True)
        o2, l2 = usv.sparse_attn_fwd(q, k, v, sel, s["k_long"], return_lse=True)
        o, lse = usv.attn_combine(o1, l1, o2, l2, return_lse=True)
        out.update(o=o, lse=lse)
    elif kind == "statistic":
        sel = usv.select_blocks(scores, kept)
        o, lse = usv.sparse_attn_fwd(q, k, v, sel, kept, return_lse=True)
        marginal, entropy = usv.attn_entropy(q, k, sel, kept, lse)
        out.update(o=o, lse=lse, marginal=marginal, entropy=entropy)
    else:
        sel = usv.select_blocks(scores, kept)
        out["o"] = usv.sparse_attn_fwd(q, k, v, sel, kept)
    out.update(scores=scores, sel=sel)
    if kind == "merged":
        o = out["o"]
        B, H, m, d = o.shape
        out["y"] = usv.token_unmerge(o.permute(0, 2, 1, 3).reshape(B, m, H * d), plan.pos)
    return out


# ------------------------------------------------------------------------------------ floor of a pass
def work(case):
    """Every input read once, every output written once; the products over the pairs that count."""
    c = case
    B, H, d = c["B"], c["H"], c["d"]
    C = H * d
    n, r, m, nb, k = _sizes(c)
    flops = nbytes = 0
    if c["kind"] in ("merged", "local"):
        nd = _destinations(c)
        z, zm, plan = 2 * B * n * C, 2 * B * (n - r) * C, 2 * 4 * B * n
        nbytes += z + z + zm + plan                       # hidden states, metric, merged states, plan
        if c["kind"] == "merged":
            flops += 2 * B * (n - nd) * nd * d            # every source against every destination
            nbytes += z                                   # unmerged output (its input is o)
        else:
            flops += 2 * B * (n - nd) * min(27, nd) * d   # a window of 3 x 3 x 3 blocks
            return {"bytes": nbytes + 2 * (z + zm) + z, "flops": flops}
    qkvo = 4 * 2 * B * m * C
    lists = 4 * B * nb * (H * nb + H * max(k))            # fp32 scores and kept lists
    pairs = B * m * sum(min(x * BLOCK, m) for x in k)
    flops += 2 * B * H * nb * nb * d + 4 * pairs * d
    nbytes += qkvo + lists
    if c["kind"] in ("statistic", "branches"):
        nbytes += 4 * B * H * m
    if c["kind"] == "statistic":
        flops += 2 * pairs * d                            # the logits once more
        nbytes += 4 * B * m
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """Measured over the listed cases and eight drawn ones, two seeds each, against the same pass with its
    sums in another order (scores from the fp32 kernel without scratch, attention from the mma.sync kernel):
    outputs differ by 4e-4 to 1.1e-3 in the 2-norm (bf16 weights and outputs).  Scores that differ by 1.5e-6
    flip near-ties at the cut of the selection, none to 8 of up to 66 864 rows: up to 7e-5 of the kept
    indices and, in the rows concerned, outputs by up to 0.08 of the root mean square."""
    if case["kind"] == "local":
        return "exact"       # the plan is whole numbers, and merged rows are sums in a fixed order
    return {"rel": 5e-3, "max": 0.3, "differ": 3e-4}
