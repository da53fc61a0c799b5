"""The work this library is asked to do, as cases that can be timed and compared.

Each case is one pass of a program that serves (or prepares) a deployment-pruned multimodal transformer
layer through the public calls of `paper_2604_08971_b200.Sentry`.  The program keeps what such a program
keeps: one library context, the weights, the gate's score tables, the prepared sample tables, and its output
buffers.  Kinds of pass:

  step    the pruned layer's three operations on tensors that are at hand: head selection and sparse attention
          (gate_attend_fwd), channel selection (gate_select), the channel-compacted FFN (ffn_fwd, which
          gathers the kept columns of the weights on every call, since the selection follows the batch's
          modality masks)
  layer   the whole layer from X: both selections, the pruned Q/K/V projections, attention, the output
          projection, the FFN on its result
  ffn     the FFN alone on weights that were materialised once per modality subset (16-bit or FP8 operands)
  moe     a Sparse-MoE block whose experts are pruned inside (routing given), weights materialised once or not
  prune   deployment: the gate's perceptrons evaluated for every modality subset, one threshold over all
          layers, the per-layer counts, and one layer's FFN weights materialised for every subset

Shapes are the workloads this repository's benchmark runs (few sensor modalities, tens to thousands of tokens per
sample, d_model 64 to 768, grouped-query attention with 2 to 4 KV heads) and ragged ones between them.
"""
import math

import numpy as np
import torch

import paper_2604_08971_b200 as sentry

_DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}
_ESIZE = {"f32": 4, "bf16": 2, "f16": 2, "fp8": 1}
_C = 5   # sparsity constant of U = c * ceil(ln T), the paper's value
_CTX = []


def _sentry():
    if not _CTX:
        _CTX.append(sentry.Sentry(0))
    return _CTX[0]


def listed():
    return [
        # the smallest call: one window of 64 tokens, as an on-line recogniser sends it; latency is all that counts
        dict(name="step_bf16_1x64", kind="step", dtype="bf16", B=1, lengths="22,21,21", masks="cycle", D=256, Hq=8, Hk=2,
             d=32, F=1024, k_h=4, k_c=512, table="arranged"),
        # the fp32 layer people debug and validate with, from X to Y
        dict(name="layer_f32_tiny", kind="layer", dtype="f32", B=2, lengths="16,16", masks="all", D=64, Hq=4, Hk=2, d=16,
             F=256, k_h=3, k_c=128, table="rows"),
        # wearable activity recognition: many short windows, sensors dropping out at random
        dict(name="step_bf16_wearable", kind="step", dtype="bf16", B=256, lengths="64,64,64", masks="dropout", D=128, Hq=8,
             Hk=2, d=16, F=512, k_h=4, k_c=256, table="arranged"),
        # physiological long windows in IEEE half, every sensor present, sample tables as they are generated
        dict(name="step_f16_physio", kind="step", dtype="f16", B=64, lengths="256,256,256,256", masks="all", D=256, Hq=8, Hk=2,
             d=32, F=1024, k_h=4, k_c=512, table="rows"),
        # the full encoder layer from X to Y, each of the three modality subsets a third of the batch
        dict(name="layer_bf16_full", kind="layer", dtype="bf16", B=128, lengths="256,256", masks="thirds", D=384, Hq=12, Hk=4,
             d=32, F=1536, k_h=7, k_c=614, table="arranged"),
        # few long sequences: K and V of a head group no longer fit in one SM
        dict(name="step_bf16_16x4096", kind="step", dtype="bf16", B=16, lengths="1366,1365,1365", masks="cycle", D=256, Hq=8,
             Hk=2, d=32, F=1024, k_h=4, k_c=512, table="columns"),
        # a server's ordinary batch of middle-sized sequences
        dict(name="step_bf16_256x1024", kind="step", dtype="bf16", B=256, lengths="342,341,341", masks="cycle", D=256, Hq=8,
             Hk=2, d=32, F=1024, k_h=4, k_c=512, table="arranged"),
        # the largest: off-line scoring of a recording, thousands of windows at once
        dict(name="step_bf16_4096x256", kind="step", dtype="bf16", B=4096, lengths="86,85,85", masks="cycle", D=256, Hq=8, Hk=2,
             d=32, F=1024, k_h=4, k_c=512, table="arranged"),
        # a base-size encoder's width (d_model 768, head dimension 64) on ragged modalities and budgets
        dict(name="step_bf16_768_ragged", kind="step", dtype="bf16", B=8, lengths="211,97,340", masks="dropout", D=768, Hq=12,
             Hk=4, d=64, F=3072, k_h=7, k_c=1229, table="rows"),
        # the FFN in FP8 arithmetic on weights materialised once per subset
        dict(name="ffn_fp8_full", kind="ffn", dtype="fp8", B=128, lengths="256,256", masks="thirds", D=384, F=1536, k_c=614),
        # a pruned Sparse-MoE block, top-2 routing of skewed popularity
        dict(name="moe_bf16_top2", kind="moe", dtype="bf16", N=32768, D=256, F=1024, E=8, top_k=2, k_c=512, packed=True),
        # deployment: four layers' channels ranked together for every subset of three sensors, one layer's weights packed
        dict(name="prune_bf16_4layers", kind="prune", dtype="bf16", M=3, layers=4, D=256, F=1024, hidden=16, keep=0.5),
    ]


# ------------------------------------------------------------------------------------------ drawing

def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _split(rng, T, M):
    cuts = sorted(rng.sample(range(1, T), M - 1)) if T > M else list(range(1, M))
    return ",".join(str(b - a) for a, b in zip([0] + cuts, cuts + [max(T, M)]))


def _candidate(rng):
    kind = rng.choices(["step", "layer", "ffn", "moe", "prune"], [11, 4, 2, 2, 1])[0]
    D = rng.choice([128, 256, 256, 384, 384, 768, 192])
    F = D * rng.choice([2, 4, 4])
    k_c = max(8, int(F * rng.uniform(0.25, 0.75)))
    if kind == "prune":
        return dict(kind=kind, dtype=rng.choice(["bf16", "f16"]), M=rng.choice([2, 3, 4]), layers=rng.randint(1, 8),
                    D=rng.choice([128, 256, 384]), F=rng.choice([512, 1024, 1536]), hidden=rng.randint(4, 32),
                    keep=round(rng.uniform(0.25, 0.75), 3))
    if kind == "moe":
        D = rng.choice([128, 256, 384])
        return dict(kind=kind, dtype=rng.choice(["bf16", "f16"]), N=_log_int(rng, 64, 40000), D=D, F=D * rng.choice([2, 4]),
                    E=rng.choice([4, 8, 16]), top_k=rng.choice([1, 2, 2, 4]), k_c=max(8, int(2 * D * rng.uniform(0.25, 0.75))),
                    packed=rng.random() < 0.6)
    M = rng.choice([2, 3, 3, 4])
    T = _log_int(rng, 24, 4096)
    c = dict(kind=kind, dtype=rng.choices(["bf16", "f16", "f32"], [6, 2, 1])[0], B=_log_int(rng, 1, 4096),
             lengths=_split(rng, T, M), masks=rng.choice(["all", "dropout", "cycle"]), D=D, F=F, k_c=k_c)
    if kind == "ffn":
        c["dtype"] = rng.choice(["bf16", "f16", "fp8", "fp8"])
        c["D"] = rng.choice([128, 256, 384])
        c["F"] = c["D"] * rng.choice([2, 4])
        c["k_c"] = max(8, int(c["F"] * rng.uniform(0.25, 0.75)))
        return c
    d = {128: [16, 32], 192: [16, 32], 256: [32], 384: [32, 64], 768: [32, 64]}[D]
    c["d"] = rng.choice(d)
    c["Hk"] = rng.choice([2, 4])
    c["Hq"] = c["Hk"] * rng.choice([2, 3, 4])
    c["k_h"] = max(1, int(c["Hq"] * rng.uniform(0.25, 0.8)))
    c["table"] = rng.choice(["rows", "arranged"]) if T <= 1024 else rng.choice(["rows", "columns"])
    return c


def draw(rng):
    """One more case of the ranges above; never more work or memory than the largest listed one."""
    top = [work(c) for c in listed()]
    most_bytes, most_flops = max(w["bytes"] for w in top), max(w["flops"] for w in top)
    while True:
        c = _candidate(rng)
        w = work(c)
        if w["bytes"] > most_bytes or w["flops"] > most_flops:
            continue
        # fp32 is for validation, and long samples of it are not
        if c["dtype"] == "f32" and (c["B"] * sum(_lengths(c)) > 4096 or c["D"] > 256):
            continue
        if c["kind"] in ("step", "layer") and c["D"] not in (128, 256, 384) and c["B"] * sum(_lengths(c)) > 6000:
            continue
        if c["kind"] in ("step", "layer", "ffn") and c["B"] * sum(_lengths(c)) > 4096 * 256:
            continue
        return c


# ------------------------------------------------------------------------------------------ shapes

def _lengths(case):
    return [int(x) for x in case["lengths"].split(",")]


def _subsets(case):
    """Modality masks that occur, with the number of samples of each (expected number for random dropout)."""
    M, B = len(_lengths(case)), case["B"]
    full = (1 << M) - 1
    if case["masks"] == "all":
        return [(full, float(B))]
    if case["masks"] == "dropout":   # each modality missing with probability 0.3, never all of them
        none = 0.3 ** M
        return [(m, B * 0.7 ** bin(m).count("1") * 0.3 ** (M - bin(m).count("1")) / (1 - none)) for m in range(1, full + 1)]
    if case["masks"] == "thirds":    # equal contiguous shares of the batch
        return [(m, float(B // full + (1 if m - 1 < B % full else 0))) for m in range(1, full + 1)]
    return [(m, float(len(range(m - 1, B, full)))) for m in range(1, min(B, full) + 1)]   # cycle


def _present(case, mask):
    return sum(n for j, n in enumerate(_lengths(case)) if (mask >> j) & 1)


def _active(tv):
    return max(1, min(tv, _C * math.ceil(math.log(tv)))) if tv > 1 else 1


def work(case):
    """Bytes and operations one pass cannot do without: kept heads, kept channels and present tokens only."""
    e, kind = _ESIZE[case["dtype"]], case["kind"]
    if kind == "prune":
        S, n, M = 1 << case["M"], case["layers"] * case["F"], case["M"]
        k, lists = int(n * case["keep"]), (1 << case["M"]) - 1
        k_c = max(8, int(case["F"] * case["keep"]))
        return {"bytes": 4.0 * n * (case["hidden"] * (M + 2) + 2 + S) + 4.0 * lists * (k + case["layers"])
                + 4.0 * lists * k_c + 2.0 * case["D"] * min(case["F"], lists * k_c) * e + 2.0 * lists * k_c * case["D"] * e,
                "flops": 2.0 * S * n * case["hidden"] * (M + 1)}
    if kind == "moe":
        rows = case["N"] * case["top_k"]
        return {"bytes": 2.0 * case["N"] * case["D"] * e + 8.0 * rows + 2.0 * case["E"] * case["k_c"] * case["D"] * e,
                "flops": 4.0 * rows * case["D"] * case["k_c"]}
    subs, T, D = _subsets(case), sum(_lengths(case)), case["D"]
    tokens = sum(n * _present(case, m) for m, n in subs)
    w_cols = min(case["F"], len(subs) * case["k_c"])
    out_e = 2 if case["dtype"] == "fp8" else e
    nbytes = tokens * D * e + case["B"] * T * D * out_e + 2.0 * w_cols * D * e
    flops = 4.0 * tokens * D * case["k_c"]
    if kind == "ffn":
        return {"bytes": nbytes, "flops": flops}
    k_h, d, Hq, Hk = case["k_h"], case["d"], case["Hq"], case["Hk"]
    r = Hq // Hk
    groups = Hk * (1 - (math.comb(Hq - r, k_h) if Hq - r >= k_h else 0) / math.comb(Hq, k_h))
    table = {_present(case, m): _present(case, m) * _active(_present(case, m)) for m, _ in subs}
    nbytes += 4.0 * sum(table.values())
    if kind == "step":   # Q, K, V are inputs
        nbytes += tokens * (k_h + 2 * groups) * d * e
    nbytes += case["B"] * k_h * T * d * e
    flops += sum(n * _present(case, m) * (6.0 * _active(_present(case, m)) * d * k_h + groups * d) for m, n in subs)
    if kind == "layer":
        nbytes += tokens * D * e + case["B"] * T * D * e + (2 * Hq + 2 * Hk) * d * D * e   # H, the output projection's result
        flops += 2.0 * tokens * D * d * (2 * k_h + 2 * groups)
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    if case["dtype"] == "f32":
        return {"rel": 1e-5, "max": 1e-3}      # 32-bit sums in another order
    if case["kind"] == "prune":
        return {"rel": 1e-5, "max": 1e-3}      # the logits; the kept lists are whole numbers and exact
    return {"rel": 1e-2, "max": 0.3}           # 16-bit results; FP8 hidden values may round to a neighbouring code


# ------------------------------------------------------------------------------------------ inputs

class _Draw:
    """Seeded tensors on the GPU."""

    def __init__(self, seed):
        self.gen = torch.Generator(device="cuda")
        self.gen.manual_seed(seed)
        self.rng = np.random.default_rng(seed)

    def normal(self, shape, std, dtype):
        x = torch.randn(shape, generator=self.gen, device="cuda", dtype=torch.float32)
        return x.mul_(std).to(dtype)

    def kept(self, rows, n, k):
        """k of n indices per row, ascending."""
        u = torch.rand((rows, n), generator=self.gen, device="cuda")
        return u.topk(k, dim=1, largest=False).indices.sort(dim=1).values.to(torch.int32).contiguous()


def _masks(case, rng):
    B, subs = case["B"], _subsets(case)
    if case["masks"] == "dropout":
        p = np.array([n for _, n in subs])
        return rng.choice([m for m, _ in subs], size=B, p=p / p.sum()).astype(np.int32)
    if case["masks"] == "thirds":
        return np.concatenate([np.full(int(n), m, np.int32) for m, n in subs])
    return np.array([subs[b % len(subs)][0] for b in range(B)], np.int32)


def _sample_tables(case, draw_, ids, sn):
    """Per subset, the sampled key positions of every query ([T_v, U] int32); subsets of one length share a table."""
    M = len(_lengths(case))
    offsets, parts, at, pos = np.full(1 << M, -1, np.int64), [], {}, 0
    for m, _ in _subsets(case):
        tv = _present(case, m)
        if tv not in at:
            t = draw_.kept(tv, tv, sentry.num_active_queries(tv, _C))
            parts.append((t.t() if case["table"] == "columns" else t).reshape(-1))
            at[tv] = pos
            pos += t.numel()
        offsets[m] = at[tv]
    table, offsets = torch.cat(parts).contiguous(), torch.from_numpy(offsets).cuda()
    if case["table"] == "arranged":
        table = sn.sample_table_arrange(ids, table, offsets, c=_C)
    return table, offsets


def _batch(case, q, s):
    """Masks, token ids and the kept-list number of every sample."""
    masks, subs = _masks(case, q.rng), [m for m, _ in _subsets(case)]
    number = {m: i for i, m in enumerate(subs)}
    s["ids"] = torch.from_numpy(np.repeat(np.arange(len(_lengths(case))), _lengths(case)).astype(np.int32)).cuda()
    s["masks"] = torch.from_numpy(masks).cuda()
    s["subsets"] = torch.tensor(subs, dtype=torch.int32, device="cuda")
    s["list_of"] = torch.tensor([number[int(m)] for m in masks], dtype=torch.int32, device="cuda")


def prepare(case, seed):
    sn, q, kind = _sentry(), _Draw(seed), case["kind"]
    s = {"case": case, "sn": sn}
    D, F = case["D"], case["F"]
    dt = _DTYPES.get(case["dtype"])
    if kind == "prune":
        n, M, h = case["layers"] * F, case["M"], case["hidden"]
        s["offsets"] = torch.arange(0, n + 1, F, dtype=torch.int32, device="cuda")
        s["zeta"], s["gamma"] = q.normal((n,), 1.0, torch.float32), q.normal((case["layers"],), 1.0, torch.float32)
        s["G1"], s["g1"] = q.normal((n, h, M), 0.5, torch.float32), q.normal((n, h), 1.0, torch.float32)
        s["G2"], s["g2"] = q.normal((n, h), 0.5, torch.float32), q.normal((n,), 1.0, torch.float32)
        s["masks"] = torch.arange(1, 1 << M, dtype=torch.int32, device="cuda")
        s["scores"] = q.normal((1 << M, F), 1.0, torch.float32)
        s["W1"], s["W2"] = q.normal((D, F), 0.02, dt), q.normal((F, D), 0.02, dt)
        return s
    if kind == "moe":
        N, E, k = case["N"], case["E"], case["top_k"]
        s["X"] = q.normal((N, D), 1.0, dt)
        W1, W2, kept = q.normal((E, D, F), 0.05, dt), q.normal((E, F, D), 0.05, dt), q.kept(E, F, case["k_c"])
        # expert e is as popular as 1 / (e + 1); k distinct experts a token by the Gumbel rule
        pop = torch.from_numpy(np.log(1.0 / (1 + q.rng.permutation(E)))).float().cuda()
        u = torch.rand((N, E), generator=q.gen, device="cuda").clamp_(1e-9, 1 - 1e-7)
        s["ids"] = (pop - torch.log(-torch.log(u))).topk(k, dim=1).indices.to(torch.int32).contiguous()
        w = -torch.log(torch.rand((N, k), generator=q.gen, device="cuda").clamp_(1e-9, 1))
        s["w"] = (w / w.sum(dim=1, keepdim=True)).contiguous()
        s["weights"] = dict(packed=sn.moe_prepack(W1, W2, kept), F=F, E=E, k_c=case["k_c"]) if case["packed"] else \
            dict(W1=W1, W2=W2, kept_channels=kept)
        s["Y"] = torch.empty_like(s["X"])
        return s
    B, T = case["B"], sum(_lengths(case))
    _batch(case, q, s)
    if kind == "ffn":
        kept = q.kept(len(s["subsets"]), F, case["k_c"])
        s["Y"] = torch.empty((B, T, D), dtype=dt or torch.bfloat16, device="cuda")
        if case["dtype"] == "fp8":
            # per-tensor scales as a calibration leaves them: the largest value at e4m3's 448 (normal draws reach about 5 sigma)
            def codes(shape, std):
                return (q.normal(shape, 448 / 5.0, torch.float32).clamp_(-448, 448).to(torch.float8_e4m3fn).view(torch.uint8),
                        5.0 * std / 448)
            (s["X"], sx), (W1, s1), (W2, s2) = codes((B, T, D), 1.0), codes((D, F), 0.02), codes((F, D), 0.02)
            s["packed"] = sn.ffn_prepack_e4m3(W1, W2, kept)
            s["scales"] = (sx, s1, s2, 5.0 * 0.02 * math.sqrt(D) / 448)
        else:
            s["X"] = q.normal((B, T, D), 1.0, dt)
            s["packed"] = sn.ffn_prepack(q.normal((D, F), 0.02, dt), q.normal((F, D), 0.02, dt), kept)
        return s
    Hq, Hk, d, k_h = case["Hq"], case["Hk"], case["d"], case["k_h"]
    S = 1 << len(_lengths(case))
    s["head_scores"], s["channel_scores"] = q.normal((S, Hq), 1.0, torch.float32), q.normal((S, F), 1.0, torch.float32)
    s["table"], s["table_offsets"] = _sample_tables(case, q, s["ids"], sn)
    s["mode"] = 0 if case["table"] == "rows" else 2
    s["X"] = q.normal((B, T, D), 1.0, dt)
    s["W1"], s["W2"] = q.normal((D, F), 0.02, dt), q.normal((F, D), 0.02, dt)
    if kind == "layer":
        s["WQ"], s["WO"] = q.normal((D, Hq * d), D ** -0.5, dt), q.normal((Hq * d, D), (k_h * d) ** -0.5, dt)
        s["WK"], s["WV"] = q.normal((D, Hk * d), D ** -0.5, dt), q.normal((D, Hk * d), D ** -0.5, dt)
        new = lambda H: torch.empty((B, H, T, d), dtype=dt, device="cuda")
        s["Q"], s["K"], s["V"], s["H"] = new(Hq), new(Hk), new(Hk), torch.empty_like(s["X"])
    else:
        s["Q"], s["K"], s["V"] = (q.normal((B, H, T, d), 1.0, dt) for H in (Hq, Hk, Hk))
    s["O"], s["Y"] = torch.empty((B, k_h, T, d), dtype=dt, device="cuda"), torch.empty_like(s["X"])
    s["kept_h"] = torch.empty((B, k_h), dtype=torch.int32, device="cuda")
    s["kept_c"] = torch.empty((len(s["subsets"]), case["k_c"]), dtype=torch.int32, device="cuda")
    return s


# ------------------------------------------------------------------------------------------ one pass

def run(s):
    case, sn, kind = s["case"], s["sn"], s["case"]["kind"]
    if kind == "step":
        sn.gate_attend_fwd(s["head_scores"], case["k_h"], s["Q"], s["K"], s["V"], s["ids"], s["masks"], s["table"],
                           s["table_offsets"], c=_C, score_mode=s["mode"], O=s["O"], kept_heads=s["kept_h"])
        sn.gate_select(s["channel_scores"], s["subsets"], case["k_c"], kept=s["kept_c"])
        sn.ffn_fwd(s["X"], s["W1"], s["W2"], s["kept_c"], s["list_of"], s["ids"], s["masks"], Y=s["Y"])
        return {"O": s["O"], "Y": s["Y"], "kept_heads": s["kept_h"], "kept_channels": s["kept_c"]}
    if kind == "layer":
        sn.gate_select_multi([(s["head_scores"], s["masks"], case["k_h"], 0, s["kept_h"]),
                              (s["channel_scores"], s["subsets"], case["k_c"], 0, s["kept_c"])])
        sn.project_qkv(s["X"], s["WQ"], s["WK"], s["WV"], s["kept_h"], s["ids"], s["masks"], case["Hq"], case["Hk"], case["d"],
                       Q=s["Q"], K=s["K"], V=s["V"])
        sn.attend_fwd(s["Q"], s["K"], s["V"], s["kept_h"], s["ids"], s["masks"], s["table"], s["table_offsets"], c=_C,
                      score_mode=s["mode"], O=s["O"])
        sn.project_out(s["O"], s["WO"], s["kept_h"], s["ids"], s["masks"], case["Hq"], out=s["H"])
        sn.ffn_fwd(s["H"], s["W1"], s["W2"], s["kept_c"], s["list_of"], s["ids"], s["masks"], Y=s["Y"])
        return {"O": s["O"], "H": s["H"], "Y": s["Y"], "kept_heads": s["kept_h"], "kept_channels": s["kept_c"]}
    if kind == "ffn":
        n_lists = len(s["subsets"])
        if case["dtype"] == "fp8":
            return sn.ffn_fwd_fp8(s["X"], s["packed"], case["F"], case["k_c"], n_lists, *s["scales"],
                                  list_of_sample=s["list_of"], token_modality_ids=s["ids"], masks=s["masks"], Y=s["Y"])
        return sn.ffn_fwd_packed(s["X"], s["packed"], case["F"], case["k_c"], n_lists, s["list_of"], s["ids"], s["masks"],
                                 Y=s["Y"])
    if kind == "moe":
        return sn.moe_ffn_fwd(s["X"], s["ids"], s["w"], Y=s["Y"], **s["weights"])
    logits = sn.gate_eval(s["offsets"], s["zeta"], s["gamma"], s["G1"], s["g1"], s["G2"], s["g2"])
    kept = sn.gate_select(logits, s["masks"], int(logits.shape[1] * case["keep"]))
    counts = sn.gate_layer_counts(kept, s["offsets"])
    lists = sn.gate_select(s["scores"], s["masks"], max(8, int(case["F"] * case["keep"])))
    packed = sn.ffn_prepack(s["W1"], s["W2"], lists)
    return {"logits": logits, "kept": kept, "counts": counts, "lists": lists,
            "packed": packed.view(torch.int16)}
