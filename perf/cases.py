"""The work that a user of this package has it do, as cases that can be timed and whose outputs can be compared.

One pass is one layer's prefill attention through the public calls: statistics of the key blocks, block selection and
sparse attention over the selected blocks (kind "layer"); selection and attention of one query chunk of a longer
sequence, as a chunked-prefill engine issues them (kind "chunk"); a batch of prompts of different lengths packed along
the token axis (kind "varlen"); and dense causal attention, the density-1 form of the attention call (kind "dense").
Inputs follow the recipe of synth.py (clustered keys, planted needles, coherent query blocks), drawn on the GPU.
"""
import math

import torch

from paper_2609_20971_b200 import (alloc_stats, rbs_block_stats, rbs_select, rbs_select_chunk, rbs_sparse_prefill,
                                   rbs_sparse_prefill_chunk, workspace_bytes)
from paper_2609_20971_b200.binding import RBS_OP_SELECT, RBS_OP_SPARSE_PREFILL, RbsShape, rbs_prefill_varlen

HEAD_DIM = 128
# (alpha_base, alpha_rescue): the default thresholds and the two alternatives of the sensitivity table
ALPHAS = ((0.22, 0.18), (0.16, 0.24), (0.24, 0.16))


def _case(kind, n, hq, hkv, block, name=None, **more):
    c = {"kind": kind, "n": n, "hq": hq, "hkv": hkv, "block": block, "alpha": 0, "sigma_ln": 0.0}
    c.update(more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the tiny configuration: one head, 4K tokens, blocks of 64 (latency of the three calls)
        _case("layer", 4096, 1, 1, 64, "layer_4k_1h_b64"),
        # a short prompt of odd length at the 32-head layer shape: the common request of a serving engine
        _case("layer", 1003, 32, 4, 128, "layer_1003_32h_b128"),
        # an ordinary long prompt
        _case("layer", 8192, 32, 4, 128, "layer_8k_32h_b128"),
        # five query heads per KV head, ragged length, log-normal key norms
        _case("layer", 16301, 40, 8, 128, "layer_16301_40h_b128", sigma_ln=0.5),
        # the 32K and 64K configurations of the 32-head layer shape (64K: log-normal key norms, here of ragged length)
        _case("layer", 32768, 32, 4, 128, "layer_32k_32h_b128"),
        _case("layer", 65451, 32, 4, 128, "layer_65451_32h_b128", sigma_ln=0.5),
        # the headline configuration
        _case("layer", 131072, 32, 4, 128, "layer_128k_32h_b128"),
        # the block-size sweep of the 64-head layer shape
        _case("layer", 131072, 64, 8, 64, "layer_128k_64h_b64"),
        _case("layer", 131072, 64, 8, 256, "layer_128k_64h_b256"),
        # chunked prefill: the last 8K tokens of a 128K prompt
        _case("chunk", 131072, 32, 4, 128, "chunk_8k_of_128k_32h_b128", start=960, tokens=8192),
        # a serving batch: prompts of different lengths packed back to back
        _case("varlen", 0, 32, 4, 128, "varlen_12_32h_b128",
              lens="512,1003,3000,777,2048,9001,333,1500,4096,640,16000,1234"),
        # dense attention, the baseline of every comparison
        _case("dense", 32768, 32, 4, 128, "dense_32k_32h"),
    ]


def draw(rng):
    def length(lo, hi):
        n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
        return n if rng.random() < 0.6 else max(lo, n // 256 * 256)      # odd lengths and round ones
    kind = rng.choice(("layer", "layer", "layer", "layer", "chunk", "chunk", "varlen", "dense"))
    block = rng.choice((64, 128, 128, 128, 256))
    hq, hkv = rng.choice(((1, 1), (4, 2), (8, 2), (16, 16), (40, 8), (32, 4), (32, 4), (32, 4), (64, 8)))
    alpha, sigma_ln = rng.randrange(len(ALPHAS)), rng.choice((0.0, 0.0, 0.5))
    if kind == "varlen":
        lens = [length(200, 16384) for _ in range(rng.randint(2, 24))]
        return _case(kind, 0, hq, hkv, block, alpha=alpha, sigma_ln=sigma_ln, lens=",".join(str(x) for x in lens))
    if kind == "dense":
        return _case(kind, length(500, 32768), hq, hkv, block)
    n = length(500, 131072)
    if kind == "chunk":
        n = max(n, 2 * block)
        m = (n + block - 1) // block
        tokens = rng.choice((2048, 4096, 8192)) // block
        start = rng.randrange(m)
        return _case(kind, n, hq, hkv, block, alpha=alpha, sigma_ln=sigma_ln, start=start,
                     tokens=min(n, (start + tokens) * block) - start * block)
    return _case(kind, n, hq, hkv, block, alpha=alpha, sigma_ln=sigma_ln)


def _inputs(n, hq, hkv, block, sigma_ln, gen):
    """One prompt's Q [1, n, hq, d], K and V [1, n, hkv, d] in bf16, by the recipe of synth.py."""
    dev, d = torch.device("cuda"), HEAD_DIM
    m, g = (n + block - 1) // block, hq // hkv

    def randn(*shape):
        return torch.randn(*shape, generator=gen, dtype=torch.float32, device=dev)

    q = torch.empty(m * block, hq, d, dtype=torch.bfloat16, device=dev)
    for h in range(hq):      # head by head: the fp32 intermediates of a whole 64-head layer would take 8 GB
        q[:, h] = (randn(m, block, d) + randn(m, 1, d)).view(m * block, d)
    v = torch.empty(m * block, hkv, d, dtype=torch.bfloat16, device=dev)
    k = torch.empty_like(v)
    for h in range(hkv):
        v[:, h] = randn(m * block, d)
        sigma = 0.1 + 0.9 * torch.rand(1, generator=gen, device=dev)
        x = randn(m, 1, d) + sigma * randn(m, block, d)
        if sigma_ln > 0:
            x = x * torch.exp(sigma_ln * randn(m, block, 1))
        # needles: a tenth of the blocks get one key along the mean of a later query block of one head of the group
        b = torch.arange(m, device=dev)
        has = torch.rand(m, generator=gen, device=dev) < 0.1
        pos = torch.randint(0, block, (m,), generator=gen, device=dev)
        later = torch.clamp(b + torch.floor(torch.rand(m, generator=gen, device=dev) * (m - b)).long(), max=m - 1)
        head = h * g + torch.randint(0, g, (m,), generator=gen, device=dev)
        mean = torch.stack([q[:, h * g + i].view(m, block, d).float().mean(1) for i in range(g)])      # [g, m, d]
        u = mean[head - h * g, later]
        u = u / u.norm(dim=1, keepdim=True).clamp_min(1e-12)
        x[b, pos] = torch.where(has[:, None], 1.5 * math.sqrt(d) * u, x[b, pos])
        k[:, h] = x.view(m * block, d)
    return q[:n].unsqueeze(0).contiguous(), k[:n].unsqueeze(0).contiguous(), v[:n].unsqueeze(0).contiguous()


def _lens(case):
    return [int(x) for x in case["lens"].split(",")]


def prepare(case, seed):
    """Inputs, and the buffers that an engine keeps from layer to layer: statistics, mask, density, workspaces, output."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    kind, n, hq, hkv, block = (case[k] for k in ("kind", "n", "hq", "hkv", "block"))
    dev = torch.device("cuda")
    s = {"case": case, "alphas": ALPHAS[case["alpha"]]}
    if kind == "varlen":
        parts = [_inputs(x, hq, hkv, block, case["sigma_ln"], gen) for x in _lens(case)]
        s["q"], s["k"], s["v"] = (torch.cat([p[i][0] for p in parts]) for i in range(3))
        cu = [0]
        for x in _lens(case):
            cu.append(cu[-1] + x)
        s["cu"], s["out"] = cu, torch.empty_like(s["q"])
        return s
    q, k, v = _inputs(n, hq, hkv, block, case["sigma_ln"], gen)
    s.update(k=k, v=v)
    m = (n + block - 1) // block
    nq, mq = n, m
    if kind == "chunk":
        t0 = case["start"] * block
        nq = case["tokens"]
        mq = (nq + block - 1) // block
        q = q[:, t0:t0 + nq].contiguous()
    s.update(q=q, out=torch.empty_like(q))
    if kind == "dense":
        return s
    shape = RbsShape(1, n, hq, hkv, HEAD_DIM, block)
    s["stats"] = alloc_stats(k, block)
    s["mask"] = torch.empty(1, hq, mq, (m + 31) // 32, dtype=torch.int32, device=dev)
    s["density"] = torch.empty(1, hq, dtype=torch.float32, device=dev)
    s["ws"] = torch.empty(max(256, workspace_bytes(RBS_OP_SELECT, shape)), dtype=torch.uint8, device=dev)
    if kind == "chunk":
        # the statistics of the prompt's keys are there: an engine takes them when the keys are written
        rbs_block_stats(k, block, s["stats"])
        s["ws_att"] = torch.empty(max(256, workspace_bytes(RBS_OP_SPARSE_PREFILL, shape)), dtype=torch.uint8, device=dev)
    return s


def run(s):
    case = s["case"]
    kind, block = case["kind"], case["block"]
    ab, ar = s["alphas"]
    if kind == "varlen":
        out, density = rbs_prefill_varlen(s["q"], s["k"], s["v"], s["cu"], block, out=s["out"], alpha_base=ab, alpha_rescue=ar)
        return {"out": out, "density": density}
    if kind == "dense":
        return {"out": rbs_sparse_prefill(s["q"], s["k"], s["v"], None, block, out=s["out"])}
    if kind == "chunk":
        mask, density = rbs_select_chunk(s["q"], s["stats"], block, case["n"], case["start"], ab, ar,
                                         mask=s["mask"], density=s["density"], workspace=s["ws"])
        out = rbs_sparse_prefill_chunk(s["q"], s["k"], s["v"], mask, block, case["start"], out=s["out"],
                                       workspace=s["ws_att"])
        return {"out": out, "mask": mask, "density": density}
    stats = rbs_block_stats(s["k"], block, s["stats"])
    mask, density = rbs_select(s["q"], stats, block, ab, ar, mask=s["mask"], density=s["density"], workspace=s["ws"])
    out = rbs_sparse_prefill(s["q"], s["k"], s["v"], mask, block, out=s["out"])
    return {"out": out, "mask": mask, "density": density, "centroid": stats.centroid, "radius": stats.radius,
            "beta": stats.beta}


def _density(m, sigma_ln):
    """Share of the causal block pairs that the selector keeps on these inputs, by the number of blocks (fitted to
    measured densities: 0.88 at 8 blocks, 0.37 at 64, 0.18 at 256, 0.080 at 1024, 0.051 at 2048; with log-normal key
    norms 0.21 at 128, 0.084 at 512)."""
    return min(1.0, 4.78 * m ** -0.59 * (0.72 if sigma_ln > 0 else 1.0))


def _sparse_work(n, hq, hkv, block, sigma_ln, first=0, rows=None):
    """Bytes and operations of selection and attention for the query blocks first .. first + rows - 1."""
    m = (n + block - 1) // block
    rows = m if rows is None else rows
    pairs = rows * first + rows * (rows + 1) / 2
    tokens = min(n, (first + rows) * block) - first * block
    flops = hq * pairs * (_density(m, sigma_ln) * 4.0 * block * block * HEAD_DIM       # attention over the kept pairs
                          + 2.0 * block * HEAD_DIM)                          # every query against every causal centroid
    # Q, O; K, V; statistics; mask
    byts = 4.0 * tokens * hq * HEAD_DIM + 4.0 * n * hkv * HEAD_DIM + 4.0 * m * hkv * (HEAD_DIM + 2) + hq * rows * m / 8
    return byts, flops


def work(case):
    kind, n, hq, hkv, block = (case[k] for k in ("kind", "n", "hq", "hkv", "block"))
    ln = case["sigma_ln"]
    if kind == "dense":
        return {"bytes": 4.0 * n * (hq + hkv) * HEAD_DIM, "flops": 2.0 * hq * float(n) * n * HEAD_DIM}
    if kind == "varlen":
        parts = [_sparse_work(x, hq, hkv, block, ln) for x in _lens(case)]
    elif kind == "chunk":
        parts = [_sparse_work(n, hq, hkv, block, ln, case["start"], (case["tokens"] + block - 1) // block)]
    else:
        parts = [_sparse_work(n, hq, hkv, block, ln)]
    return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}


def tolerance(case):
    """Outputs are bf16 from bf16 inputs, with the probabilities rounded to bf16 before the product with V: against the
    same path in 64 bits the attention output is off by 1.1e-3 to 1.9e-3 (2-norm).  A mask decision may fall the other
    way where a score lies within rounding (about 1e-5 relative) of its threshold: none of 25,000 mask words did."""
    if case["kind"] in ("dense", "varlen"):
        return {"rel": 7e-3}
    m = (case["n"] + case["block"] - 1) // case["block"]
    rows = m if case["kind"] == "layer" else (case["tokens"] + case["block"] - 1) // case["block"]
    words = case["hq"] * rows * ((m + 31) // 32)
    return {"rel": 7e-3, "differ": min(0.5, max(2e-4, 2.5 / words))}


def _exact_stats(k, block):
    """Centroids [hkv, m, d], radii and rescue coefficients [hkv, m] in 64 bits of the keys k [n, hkv, d]."""
    n = k.shape[0]
    full = n // block
    parts = [k[:full * block].double().view(full, block, *k.shape[1:])] if full else []
    if n > full * block:
        parts.append(k[full * block:].double().unsqueeze(0))
    c = torch.cat([p.mean(1) for p in parts])                                              # [m, hkv, d]
    r = torch.cat([(p - p.mean(1, keepdim=True)).norm(dim=-1).amax(1) for p in parts])     # [m, hkv]
    lo, hi = torch.quantile(r, 0.5, dim=0), torch.quantile(r, 0.9, dim=0)
    beta = torch.where(hi > lo, ((r - lo) / torch.where(hi > lo, hi - lo, torch.ones_like(hi))).clamp(0, 1), torch.zeros_like(r))
    return c.transpose(0, 1), r.t(), beta.t()


def _exact_rows(q, k, v, stats, block, first, alphas):
    """Selection and attention in 64 bits of the query tokens q [nq, hq, d] from query block `first` on: output as q,
    kept blocks [hq, rows, m].  `stats` None: dense."""
    nq, hq, d = q.shape
    n, hkv = k.shape[:2]
    m, rows = (n + block - 1) // block, (nq + block - 1) // block
    out = torch.empty(nq, hq, d, dtype=torch.float64, device=q.device)
    keep = torch.zeros(hq, rows, m, dtype=torch.bool, device=q.device)
    pos, col = torch.arange(first * block, first * block + nq, device=q.device), torch.arange(n, device=q.device)
    for h in range(hq):
        hk = h // (hq // hkv)
        qh, kh, vh = q[:, h].double() / math.sqrt(d), k[:, hk].double(), v[:, hk].double()
        for i in range(rows):
            t0, t1 = i * block, min(nq, (i + 1) * block)
            at = first + i
            nb = at + 1
            if stats is None:
                rest = kept = None
                keys, vals, cols = kh[:min(n, nb * block)], vh[:min(n, nb * block)], col[:min(n, nb * block)]
            else:
                c, r, beta = (x[hk, :nb] for x in stats)
                z = qh[t0:t1] @ c.t()
                zr = z + qh[t0:t1].norm(dim=1, keepdim=True) * (r * beta)
                sb, sr = torch.logsumexp(z, 0), torch.logsumexp(zr, 0)
                kept = (sb >= math.log(alphas[0]) + sb.max()) | (sr >= math.log(alphas[1]) + sr.max())
                kept[0] = kept[at] = True                       # the first block and the query block's own
                if at == m - 1:                                 # the sequence's last query block keeps all
                    kept[:] = True
                keep[h, i, :nb] = kept
                rest = kept.nonzero()[:, 0]
                cols = (rest[:, None] * block + torch.arange(block, device=q.device)).flatten()
                cols = cols[:cols.numel() - max(0, nb * block - n)]          # the last kept block is the query block's own
                keys, vals = kh[cols], vh[cols]
            s = qh[t0:t1] @ keys.t()
            s.masked_fill_(cols[None, :] > pos[t0:t1, None], -math.inf)
            out[t0:t1, h] = torch.softmax(s, 1) @ vals
    return out, keep


def _words(keep):
    """[hq, rows, m] kept blocks -> [1, hq, rows, words] 32-bit words, block b in bit b % 32 of word b / 32."""
    w = (keep.shape[-1] + 31) // 32
    bits = torch.nn.functional.pad(keep, (0, 32 * w - keep.shape[-1])).view(*keep.shape[:-1], w, 32).long()
    x = (bits << torch.arange(32, device=keep.device)).sum(-1)
    return torch.where(x >= 1 << 31, x - (1 << 32), x).int().unsqueeze(0)


def exact(case, seed):
    """What run() returns for these inputs, from their bf16 values on in 64 bits by the paper's formulas; None where that
    would take longer than about 20 seconds."""
    kind, n, block = case["kind"], case["n"], case["block"]
    lens = _lens(case) if kind == "varlen" else [n]
    m = sum((x + block - 1) // block for x in lens)
    if (m if kind != "chunk" else (case["tokens"] + block - 1) // block) * case["hq"] > 20000:
        return None
    s = prepare(case, seed)
    if kind == "varlen":
        outs, dens = [], []
        for t0, t1 in zip(s["cu"], s["cu"][1:]):
            q, k, v = (s[x][t0:t1] for x in "qkv")
            out, keep = _exact_rows(q, k, v, _exact_stats(k, block), block, 0, s["alphas"])
            outs.append(out)
            dens.append(keep.sum((1, 2)).double() / (keep.shape[2] * (keep.shape[2] + 1) / 2))
        return {"out": torch.cat(outs), "density": torch.stack(dens)}
    q, k, v = (s[x][0] for x in "qkv")
    if kind == "dense":
        return {"out": _exact_rows(q, k, v, None, block, 0, None)[0].unsqueeze(0)}
    c, r, beta = _exact_stats(k, block)
    first = case["start"] if kind == "chunk" else 0
    out, keep = _exact_rows(q, k, v, (c, r, beta), block, first, s["alphas"])
    rows = keep.shape[1]
    density = keep.sum((1, 2)).double() / (rows * first + rows * (rows + 1) / 2)
    res = {"out": out.unsqueeze(0), "mask": _words(keep), "density": density.unsqueeze(0)}
    if kind == "layer":
        res.update(centroid=c.unsqueeze(0), radius=r.unsqueeze(0), beta=beta.unsqueeze(0))
    return res
