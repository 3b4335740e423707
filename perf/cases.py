"""The work a program has this library do, as timed cases.

Every case goes through the package's entry points with the buffers, workspaces and weights a serving or
training program would keep.  Kinds of cases:

  step     one decode step over a merged context: merge module, rollback of the spans, attention
  merge    the merge module alone, on the few spans that one decoding step completes
  prompt   prompt compression: merge module over the prompts' spans, then the packed compressed prompts
  context  rollback of a long context's spans (keys moved verbatim or re-rotated), then attention
  layers   a serving engine's decode step, one fused call per layer
  engine   a serving engine's decode step as one cache update and one attention call per layer
  prefill  causal attention over the packed compressed prompts
  rules    prompt compression by rule matching and precomputed surrogates
  distill  alignment of teacher and student rows, soft-target cross-entropy and its gradient

Inputs are drawn on the GPU from the seed: N(0, 0.02^2) embeddings, N(0, 1) cache entries and queries,
U(+-1/sqrt(d)) linear weights, spans of 2 to 4 tokens at uniformly drawn places, pages in random order.
Sizes (lengths, how many spans) belong to the case and are only put in another order by the seed.
"""
import math
from statistics import NormalDist

import numpy as np
import torch

import paper_2609_27233_gb300 as umim

PAGE = 16
VOCAB = 128256
RULE_COUNTS = (216700, 684793, 1266080)   # 2-, 3- and 4-grams of a full rule set
BF16 = torch.bfloat16


def listed():
    return [
        # an interactive request on a small model: the shortest calls, where launches and latency count
        dict(name="tiny step", kind="step", B=1, L=512, hq=8, hkv=2, D=64, coverage=0.24, d=512, vocab=32000),
        # one layer's step for a batch of 16 requests of 4096 tokens on an 8B model
        dict(name="8B layer step", kind="step", B=16, L=4096, hq=32, hkv=8, D=128, coverage=0.3, d=4096, vocab=VOCAB),
        # the spans that a decode step of 128 sequences completes (a tenth of them)
        dict(name="decode merges", kind="merge", S=13, d=4096, h=4, vocab=VOCAB),
        # one prompt of an odd length on its way into prefill
        dict(name="one prompt", kind="prompt", B=1, L=1931, coverage=0.37, d=4096, vocab=VOCAB),
        # a batch of prompts compressed together
        dict(name="64 prompts", kind="prompt", B=64, L=2048, coverage=0.4, d=4096, vocab=VOCAB),
        # long documents whose keys keep their compressed positions (RoPE), 28 query heads
        dict(name="long context", kind="context", B=4, L=32768, hq=28, hkv=4, D=128, coverage=0.4, rope=True),
        # a loaded serving engine: 128 sequences of mixed lengths, four layers of one step
        dict(name="serving layers", kind="layers", B=128, layers=4, hq=32, hkv=8, D=128, median=1024, p=0.1),
        # a lightly loaded engine: a few short sequences, update and attention calls
        dict(name="light engine", kind="engine", B=3, layers=4, hq=32, hkv=8, D=128, median=700, p=0.3),
        # prefill of a batch of compressed prompts, one layer of an 8B model
        dict(name="prefill batch", kind="prefill", B=64, rows=1500, hq=32, hkv=8, D=128),
        # prefill of a handful of short ragged prompts on a small model
        dict(name="prefill ragged", kind="prefill", B=5, rows=347, hq=8, hkv=2, D=64),
        # prompts compressed with a full rule set and its lookup table
        dict(name="rule lookup", kind="rules", B=64, L=2048, coverage=0.4, d=4096, vocab=VOCAB, rules=1.0),
        # the distillation objective on a training batch of 8 x 512 tokens
        dict(name="distillation", kind="distill", B=8, L=512, coverage=0.4, V=VOCAB, eps=1e-8, grad=True),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["step", "step", "merge", "prompt", "context", "layers", "engine", "prefill", "prefill",
                       "rules", "distill"])
    hq, hkv, D = rng.choice([(8, 2, 64), (32, 8, 128), (28, 4, 128), (8, 8, 64), (32, 2, 128), (32, 8, 128)])
    d = rng.choice([512, 1024, 2048, 4096, 4096])
    coverage = round(rng.uniform(0.1, 0.5), 3)
    if kind == "step":
        return dict(kind=kind, B=_log_int(rng, 1, 16), L=_log_int(rng, 128, 4096), hq=hq, hkv=hkv, D=D,
                    coverage=min(coverage, 0.3), d=d, vocab=rng.choice([32000, VOCAB]))
    if kind == "merge":
        return dict(kind=kind, S=_log_int(rng, 1, 2048), d=rng.choice([512, 1024, 1536, 2048, 4096, 4096, 8192]),
                    h=rng.choice([1, 2, 4, 4, 4, 8]), vocab=32000)
    if kind == "prompt":
        return dict(kind=kind, B=_log_int(rng, 1, 48), L=_log_int(rng, 64, 2048), coverage=min(coverage, 0.4), d=d,
                    vocab=rng.choice([32000, VOCAB]))
    if kind == "context":
        return dict(kind=kind, B=_log_int(rng, 1, 4), L=_log_int(rng, 2048, 32768), hq=hq, hkv=min(hkv, 4), D=D,
                    coverage=coverage, rope=rng.random() < 0.5)
    if kind in ("layers", "engine"):
        return dict(kind=kind, B=_log_int(rng, 1, 128), layers=rng.choice([1, 2, 4]), hq=hq, hkv=hkv, D=D,
                    median=_log_int(rng, 64, 1024), p=round(rng.uniform(0.0, 0.5), 2))
    if kind == "prefill":
        return dict(kind=kind, B=_log_int(rng, 1, 48), rows=_log_int(rng, 24, 1500), hq=hq, hkv=hkv, D=D)
    if kind == "rules":
        return dict(kind=kind, B=_log_int(rng, 1, 64), L=_log_int(rng, 64, 2048), coverage=min(coverage, 0.4),
                    d=rng.choice([512, 1024, 2048]), vocab=VOCAB, rules=rng.choice([0.01, 0.1, 0.5]))
    return dict(kind="distill", B=_log_int(rng, 1, 8), L=_log_int(rng, 32, 512), coverage=min(coverage, 0.4),
                V=rng.choice([1001, 32000, 50257, VOCAB, rng.randrange(2000, VOCAB)]), eps=rng.choice([0.0, 1e-8, 1e-4]),
                grad=rng.random() < 0.8)


# ----------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------
class _Draw:
    """Seeded draws: structure from numpy, bulk tensors from a generator on the GPU."""

    def __init__(self, seed):
        self.dev = torch.device("cuda")
        self.np = np.random.Generator(np.random.PCG64(seed))
        self.gen = torch.Generator(device=self.dev)
        self.gen.manual_seed(seed)

    def normal(self, shape, std=1.0, dtype=BF16):
        out = torch.empty(shape, dtype=dtype, device=self.dev)
        flat, step = out.view(-1), 1 << 28
        for i in range(0, flat.numel(), step):
            part = flat[i:i + step]
            part.copy_(torch.randn(part.numel(), generator=self.gen, device=self.dev).mul_(std))
        return out

    def uniform(self, shape, lo, hi):
        return (torch.rand(shape, generator=self.gen, device=self.dev) * (hi - lo) + lo).to(BF16)

    def put(self, a, dtype=np.int32):
        return torch.from_numpy(np.ascontiguousarray(np.asarray(a, dtype))).to(self.dev)

    def spans(self, L, coverage):
        """Sorted, disjoint spans of 2 to 4 positions that cover about `coverage` of [0, L)."""
        want = int(round(coverage * L))
        lens = np.arange(want // 2 + 1) % 3 + 2
        lens = lens[: max(1 if L >= 4 else 0, int(np.searchsorted(np.cumsum(lens), want)))]
        lens = self.np.permutation(lens)
        S, free = len(lens), L - int(lens.sum())
        bars = np.sort(self.np.choice(free + S, size=S, replace=False)) - np.arange(S)
        return (bars + np.concatenate([[0], np.cumsum(lens)[:-1]])[:S]).astype(np.int32), lens.astype(np.int32)

    def span_lists(self, lens, coverage):
        """(offsets, start, length) over all sequences."""
        each = [self.spans(int(L), coverage) for L in lens]
        offsets = np.concatenate([[0], np.cumsum([len(s) for s, _ in each])]).astype(np.int32)
        return offsets, np.concatenate([s for s, _ in each]), np.concatenate([n for _, n in each])


def _weights(r, d, h):
    a = 1.0 / math.sqrt(d)
    return dict(w_kv=r.uniform((d, d), -a, a), b_kv=r.uniform((d,), -a, a), ln_kv_gamma=r.uniform((d,), 0.9, 1.1),
                ln_kv_beta=r.uniform((d,), -0.1, 0.1), query=r.normal((h, d // h)), w_o=r.uniform((d, d), -a, a),
                b_o=r.uniform((d,), -a, a), ln_o_gamma=r.uniform((d,), 0.9, 1.1), ln_o_beta=r.uniform((d,), -0.1, 0.1),
                d_model=d, n_heads=h, ln_eps=1e-5)


def _cache(r, lens, hq, hkv, D, layers=1, room=0):
    """A paged cache with `lens` entries (pages in random order) and queries; `room`: entries still to come."""
    lens = np.asarray(lens, np.int64)
    now, most = -(-lens // PAGE), -(-(lens + room) // PAGE)
    perm = r.np.permutation(int(most.sum()) + 1).astype(np.int32)
    table = np.full((len(lens), int(most.max())), -1, np.int32)
    for b, first in enumerate(np.cumsum(most) - most):
        table[b, :now[b]] = perm[first:first + now[b]]
    opened = [perm[first + now[b]] if L % PAGE == 0 and room else -1
              for b, (first, L) in enumerate(zip(np.cumsum(most) - most, lens))]
    return dict(table=table, lens=lens.astype(np.int32), new_pages=np.asarray(opened, np.int32),
                pool=r.normal((layers, len(perm), 2, hkv, PAGE, D)), q=r.normal((layers, len(lens), hq, D)))


def _inputs(case, seed):
    """Everything the case is computed from: tensors on the GPU, structure as numpy arrays."""
    r = _Draw(seed)
    kind, x = case["kind"], {}
    if kind in ("step", "prompt", "merge"):
        x["w"] = _weights(r, case["d"], case.get("h", 4))
        x["emb"] = r.normal((case["vocab"], case["d"]), 0.02)
    if kind == "merge":
        n = r.np.permutation(np.arange(case["S"]) % 3 + 2)
        x["offs"] = np.concatenate([[0], np.cumsum(n)]).astype(np.int32)
        x["ids"] = r.np.integers(0, case["vocab"], size=int(x["offs"][-1])).astype(np.int32)
    if kind in ("step", "context"):
        lens = [case["L"]] * case["B"]
        x["spans"] = r.span_lists(lens, case["coverage"])
        x.update(_cache(r, lens, case["hq"], case["hkv"], case["D"]))
        S = len(x["spans"][1])
        x["sk"], x["sv"] = r.normal((S, 1, case["hkv"], case["D"])), r.normal((S, 1, case["hkv"], case["D"]))
        if case.get("rope"):
            D = case["D"]
            x["freq"] = torch.from_numpy((500000.0 ** (-np.arange(0, D, 2) / D)).astype(np.float32)).to(r.dev)
    if kind == "step":
        n = x["spans"][2]
        x["offs"] = np.concatenate([[0], np.cumsum(n)]).astype(np.int32)
        x["ids"] = r.np.integers(0, case["vocab"], size=int(x["offs"][-1])).astype(np.int32)
    if kind == "prompt":
        tokens = r.np.integers(0, case["vocab"], size=(case["B"], case["L"])).astype(np.int32)
        so, ss, sn = x["spans"] = r.span_lists([case["L"]] * case["B"], case["coverage"])
        row = np.repeat(np.arange(case["B"]), np.diff(so))
        x["offs"] = np.concatenate([[0], np.cumsum(sn)]).astype(np.int32)
        inside = np.arange(int(x["offs"][-1])) - np.repeat(x["offs"][:-1], sn)
        x["tokens"], x["ids"] = tokens, tokens[np.repeat(row, sn), np.repeat(ss, sn) + inside]
    if kind in ("layers", "engine"):
        # the quantiles of a log-normal distribution, one sequence at least opening a page
        B = case["B"]
        z = np.array([NormalDist().inv_cdf((i + 0.5) / B) for i in range(B)])
        lens = np.clip(np.round(case["median"] * np.exp(z)), 16, 8 * case["median"]).astype(np.int64)
        lens[0] = (lens[0] // PAGE) * PAGE
        lens = r.np.permutation(lens)
        x.update(_cache(r, lens, case["hq"], case["hkv"], case["D"], case["layers"], room=PAGE))
        shape = (case["B"], case["layers"], case["hkv"], case["D"])
        x["nk"], x["nv"] = r.normal(shape), r.normal(shape)
        hit = r.np.permutation(np.arange(B) < round(case["p"] * B))
        x["merge_k"] = np.where(hit, r.np.integers(2, 5, size=B), 0).astype(np.int32)
        x["merge_row"] = np.where(hit, np.cumsum(hit) - 1, -1).astype(np.int32)
        rows = max(1, int(hit.sum()))
        x["sk"], x["sv"] = r.normal((rows, *shape[1:])), r.normal((rows, *shape[1:]))
    if kind == "prefill":
        lens = np.maximum(1, np.round(case["rows"] * (0.8 + 0.4 * (np.arange(case["B"]) + 0.5) / case["B"])))
        lens = r.np.permutation(lens.astype(np.int64))
        x["cu"] = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
        T = int(x["cu"][-1])
        x["q"] = r.normal((T, case["hq"], case["D"]))
        x["k"], x["v"] = r.normal((T, case["hkv"], case["D"])), r.normal((T, case["hkv"], case["D"]))
    if kind == "rules":
        V, d = case["vocab"], case["d"]
        grams, by_n = [], []
        for n, c in zip((2, 3, 4), RULE_COUNTS):
            c = max(16, int(c * case["rules"]))
            g = torch.full((c + 64, 4), -1, dtype=torch.int64, device=r.dev)
            g[:, :n] = torch.randint(0, V, (c + 64, n), generator=r.gen, device=r.dev)
            key = (g[:, 0] * V + g[:, 1]) * V + (g[:, 2] if n > 2 else 0)   # distinct keys: distinct n-grams
            key, back = torch.sort(key, stable=True)
            first = torch.ones_like(key, dtype=torch.bool)
            first[1:] = key[1:] != key[:-1]
            g = g[back[first]]
            grams.append(g[torch.randperm(len(g), generator=r.gen, device=r.dev)[:c]])
        rules = torch.cat(grams)
        order = torch.randperm(len(rules), generator=r.gen, device=r.dev)
        x["rules"] = rules[order].to(torch.int32).contiguous()
        host = x["rules"].cpu().numpy()
        by_n = [np.nonzero((host >= 0).sum(1) == n)[0] for n in (2, 3, 4)]
        tokens = r.np.integers(0, V, size=(case["B"], case["L"])).astype(np.int32)
        so, ss, sn = r.span_lists([case["L"]] * case["B"], case["coverage"])
        row = np.repeat(np.arange(case["B"]), np.diff(so))
        for n in (2, 3, 4):
            at = np.nonzero(sn == n)[0]
            which = by_n[n - 2][r.np.integers(0, len(by_n[n - 2]), size=len(at))]
            for i in range(n):
                tokens[row[at], ss[at] + i] = host[which, i]
        x["tokens"], x["planted"] = tokens, len(ss)
        x["emb"] = r.normal((V, d), 0.02)
        x["lut"] = r.normal((len(host), d), dtype=torch.float32)
    if kind == "distill":
        lens = np.asarray([case["L"]] * case["B"], np.int32)
        x["lens"], x["spans"] = lens, r.span_lists(lens, case["coverage"])
        R_T = int(lens.sum())
        ld = -(-case["V"] // 8) * 8
        x["teacher"] = r.normal((R_T, ld), 2.0)
        x["student"] = r.normal((R_T - int((x["spans"][2] - 1).sum()), ld), 2.0)
    return x, r


# ----------------------------------------------------------------------------
# what a program keeps, and one pass
# ----------------------------------------------------------------------------
def prepare(case, seed):
    x, r = _inputs(case, seed)
    kind, dev = case["kind"], r.dev
    s = dict(case=dict(case), status=umim.new_status(dev))
    i32 = lambda n, v=0: torch.full((n,), v, dtype=torch.int32, device=dev)
    for k in ("emb", "w", "pool", "q", "sk", "sv", "nk", "nv", "k", "v", "freq", "teacher", "student", "lut"):
        if k in x:
            s[k] = x[k]
    if "ids" in x:
        s["ids"], s["offs"] = r.put(x["ids"]), r.put(x["offs"])
        T, S, d = len(x["ids"]), len(x["offs"]) - 1, case["d"]
        s["z"] = torch.zeros((S, d), dtype=torch.float32, device=dev)
        s["ws_merge"] = umim.workspace(umim.umim_merge_spans_workspace_size(T, S, d), dev)
    if "spans" in x:
        s["so"], s["ss"], s["sn"] = (r.put(a) for a in x["spans"])
        S = len(x["spans"][1])
    if "table" in x:
        # the scheduler's tables, lengths last, sent whole before each step
        s["tables0"] = torch.cat([r.put(x["table"]).view(-1), r.put(x["lens"])])
        s["tables"] = s["tables0"].clone()
        B, pages = x["table"].shape
        s["bt"], s["lens"] = s["tables"][:B * pages].view(B, pages), s["tables"][B * pages:]
        s["out"] = torch.empty_like(s["q"])
    if kind in ("step", "context"):
        s["q"], s["out"] = s["q"][0], s["out"][0]
        s["freed"] = i32(B * pages, -2)
        s["ws_roll"] = umim.workspace(umim.umim_kv_rollback_workspace_size(B, S, pages, 1, case["hkv"], case["D"]), dev)
    if kind in ("step", "context", "engine"):
        s["ws_attn"] = umim.workspace(umim.umim_decode_attention_workspace_size(B, case["hq"], case["hkv"], case["D"]),
                                      dev)
    if kind in ("layers", "engine"):
        for k in ("new_pages", "merge_k", "merge_row"):
            s[k] = r.put(x[k])
        s["released"] = i32(B, -2)
    if kind == "layers":
        s["sk"], s["sv"] = ([t[:, l].contiguous() for l in range(case["layers"])] for t in (s["sk"], s["sv"]))
        s["ws_step"] = umim.workspace(umim.umim_decode_layer_step_workspace_size(B, case["hkv"], case["D"]), dev)
    if kind in ("prompt", "rules"):
        s["tokens"] = r.put(x["tokens"])
        rows = case["B"] * case["L"]
        s["embeds"] = torch.zeros((rows, case["d"]), dtype=BF16, device=dev)
        s["positions"], s["cu"] = i32(rows), i32(case["B"] + 1)
        cap = S if kind == "prompt" else max(1, case["B"] * (case["L"] // 2))
        s["ws_build"] = umim.workspace(umim.umim_build_compressed_workspace_size(case["B"], cap), dev)
    if kind == "rules":
        s["table"] = umim.umim_rules_build(x["rules"], dev_status=s["status"])
        s["match"] = dict(span_offsets=i32(case["B"] + 1), span_start=i32(cap), span_len=i32(cap), span_rule=i32(cap),
                          merge_token_ids=None, merge_offsets=None)
        s["z"] = torch.zeros((cap, case["d"]), dtype=torch.float32, device=dev)
        s["ws_match"] = umim.workspace(umim.umim_match_prompts_workspace_size(case["B"], case["L"]), dev)
    if kind == "prefill":
        s["cu"], s["out"] = r.put(x["cu"]), torch.empty_like(s["q"])
        s["ws"] = umim.workspace(umim.umim_prefill_attention_workspace_size(case["B"], s["q"].shape[0], case["hkv"],
                                                                            case["D"]), dev)
    if kind == "distill":
        s["seq_lens"] = r.put(x["lens"])
        R_S = s["student"].shape[0]
        s["pairs"] = dict(pair_offsets=i32(case["B"] + 1), teacher_rows=i32(R_S), student_rows=i32(R_S),
                          student_cu=i32(case["B"] + 1))
        s["n"] = s["pairs"]["pair_offsets"][case["B"]:]
        s["loss"] = torch.zeros(1, device=dev)
        s["pair_loss"] = torch.zeros(R_S, device=dev)
        s["grad"] = torch.zeros_like(s["student"]) if case["grad"] else None
        s["ws_align"] = umim.workspace(umim.umim_distill_align_workspace_size(case["B"], S), dev)
        s["ws_ce"] = umim.workspace(umim.umim_distill_soft_ce_workspace_size(R_S, R_S), dev)
    return s


def run(s):
    case, st = s["case"], s["status"]
    kind, out = case["kind"], []
    if kind in ("step", "merge", "prompt"):
        umim.umim_merge_spans(s["emb"], s["ids"], s["offs"], s["w"], surrogates=s["z"], workspace_buf=s["ws_merge"],
                              dev_status=st)
        out.append(s["z"])
    if kind in ("step", "context"):
        s["tables"].copy_(s["tables0"])
        umim.umim_kv_rollback(s["pool"], s["bt"], s["lens"], s["so"], s["ss"], s["sn"], s["sk"], s["sv"],
                              freed_pages=s["freed"], workspace_buf=s["ws_roll"], dev_status=st,
                              rope_inv_freq=s.get("freq"))
        umim.umim_decode_attention(s["q"], s["pool"], 0, s["bt"], s["lens"], out=s["out"], workspace_buf=s["ws_attn"],
                                   dev_status=st)
        out += [s["out"], s["bt"], s["lens"], s["freed"], s["pool"]]
    if kind == "layers":
        s["tables"].copy_(s["tables0"])
        last = case["layers"] - 1
        for l in range(last + 1):
            umim.umim_decode_layer_step(s["q"][l], s["pool"], l, s["bt"], s["lens"], s["nk"][:, l], s["nv"][:, l],
                                        new_pages=s["new_pages"], merge_k=s["merge_k"], merge_row=s["merge_row"],
                                        surrogate_k=s["sk"][l], surrogate_v=s["sv"][l], commit=l == last,
                                        released=s["released"], out=s["out"][l], workspace_buf=s["ws_step"],
                                        dev_status=st)
    if kind == "engine":
        s["tables"].copy_(s["tables0"])
        umim.umim_decode_append_merge(s["pool"], s["bt"], s["lens"], s["nk"], s["nv"], new_pages=s["new_pages"],
                                      merge_k=s["merge_k"], merge_row=s["merge_row"], surrogate_k=s["sk"],
                                      surrogate_v=s["sv"], released=s["released"], dev_status=st)
        for l in range(case["layers"]):
            umim.umim_decode_attention(s["q"][l], s["pool"], l, s["bt"], s["lens"], out=s["out"][l],
                                       workspace_buf=s["ws_attn"], dev_status=st)
    if kind in ("layers", "engine"):
        out += [s["out"], s["bt"], s["lens"], s["released"], s["pool"]]
    if kind == "rules":
        m = umim.umim_match_prompts(s["table"], s["tokens"], out=s["match"], workspace_buf=s["ws_match"], dev_status=st)
        umim.umim_lookup_surrogates(s["lut"], m["span_rule"], n_dev=m["span_offsets"][case["B"]:], out=s["z"],
                                    dev_status=st)
        s["so"], s["ss"], s["sn"] = m["span_offsets"], m["span_start"], m["span_len"]
        out += [s["so"], s["ss"], s["sn"], m["span_rule"], s["z"]]
    if kind in ("prompt", "rules"):
        umim.umim_build_compressed(s["emb"], s["tokens"], s["so"], s["ss"], s["sn"], s["z"], out_embeds=s["embeds"],
                                   position_ids=s["positions"], cu_seqlens=s["cu"], workspace_buf=s["ws_build"],
                                   dev_status=st)
        out += [s["embeds"], s["positions"], s["cu"]]
    if kind == "prefill":
        umim.umim_prefill_attention(s["q"], s["k"], s["v"], s["cu"], out=s["out"], workspace_buf=s["ws"], dev_status=st)
        out.append(s["out"])
    if kind == "distill":
        p = umim.umim_distill_align(s["seq_lens"], s["so"], s["ss"], s["sn"], s["student"].shape[0], out=s["pairs"],
                                    workspace_buf=s["ws_align"], dev_status=st)
        umim.umim_distill_soft_ce(s["teacher"], s["student"], p["teacher_rows"], p["student_rows"], n_pairs=s["n"],
                                  vocab=case["V"], eps=case["eps"], with_grad=case["grad"], loss=s["loss"],
                                  pair_loss=s["pair_loss"], grad=s["grad"], workspace_buf=s["ws_ce"], dev_status=st)
        out += [s["loss"], s["pair_loss"], p["pair_offsets"], p["teacher_rows"], p["student_rows"], p["student_cu"]]
        out += [s["grad"]] if case["grad"] else []
    out.append(st)
    return out


# ----------------------------------------------------------------------------
# what a pass cannot do without
# ----------------------------------------------------------------------------
def work(case):
    """Expected sizes (3 tokens a span, every length at its mean): each input read once, each output written once."""
    kind, B, nbytes, flops = case["kind"], case.get("B", 1), 0.0, 0.0
    L = case.get("L", 0)
    S = case["S"] if kind == "merge" else B * L * case.get("coverage", 0) / 3
    if kind in ("step", "merge", "prompt"):
        d = case["d"]
        nbytes += 3 * S * d * 2 + 2 * d * d * 2 + S * d * 4
        flops += 2 * (3 * S + S) * d * d
    if kind in ("step", "context"):
        entry = 2 * case["hkv"] * case["D"] * 2
        left = B * L - 2 * S                      # entries after the rollback
        nbytes += 2 * left * entry                # moved entries and surrogates, read and written
        nbytes += left * entry + 4 * B * case["hq"] * case["D"]
        flops += 4 * left * case["hq"] * case["D"]
    if kind in ("layers", "engine"):
        entry = 2 * case["hkv"] * case["D"] * 2
        mean = 1.5 * case["median"]               # of the clipped log-normal lengths
        nbytes += case["layers"] * B * ((mean + 2) * entry + 4 * case["hq"] * case["D"])
        flops += case["layers"] * B * 4 * mean * case["hq"] * case["D"]
    if kind == "prompt":
        nbytes += (B * L - 2 * S) * case["d"] * 2 + (B * L - 3 * S) * case["d"] * 2 + S * case["d"] * 4
    if kind == "rules":
        nbytes += 2 * S * case["d"] * 4 + (B * L - 2 * S) * case["d"] * 2 + (B * L - 3 * S) * case["d"] * 2
        nbytes += S * case["d"] * 4 + B * L * 4
    if kind == "prefill":
        T, n = B * case["rows"], case["rows"]
        nbytes += T * (2 * case["hq"] + 2 * case["hkv"]) * case["D"] * 2
        flops += 4 * T * (n * 1.013 + 1) / 2 * case["hq"] * case["D"]
    if kind == "distill":
        rows = B * L - 2 * S
        nbytes += rows * case["V"] * 2 * (3 if case["grad"] else 2)
        flops += rows * case["V"] * 20
    return dict(bytes=nbytes, flops=flops)


def tolerance(case):
    """Outputs in bf16 carry its rounding (1.7e-3 in the 2-norm); surrogates go through 16-bit tensor-core operands."""
    return {"step": {"rel": 7e-3, "max": 0.1}, "context": {"rel": 7e-3, "max": 0.1}, "layers": {"rel": 7e-3, "max": 0.1},
            "engine": {"rel": 7e-3, "max": 0.1}, "prefill": {"rel": 7e-3, "max": 0.1},
            "merge": {"rel": 1.5e-3, "max": 0.05}, "prompt": {"rel": 7e-3, "max": 0.1},
            "distill": {"rel": 7e-3, "max": 0.05}}.get(case["kind"], "exact")


# ----------------------------------------------------------------------------
# the same in 64 bits, in plain torch
# ----------------------------------------------------------------------------
def _merge64(x, case):
    w, d = x["w"], case["d"]
    h, offs = w["n_heads"], x["offs"]
    n = np.diff(offs)
    f = {k: v.double() for k, v in w.items() if isinstance(v, torch.Tensor)}
    dev = x["emb"].device
    out = torch.empty((len(n), d), dtype=torch.float64, device=dev)
    F = torch.nn.functional
    for a in range(0, len(n), 4096):
        b = min(len(n), a + 4096)
        ids = torch.from_numpy(x["ids"][offs[a]:offs[b]]).long().to(dev)
        P = F.gelu(x["emb"][ids].double() @ f["w_kv"].T + f["b_kv"])
        P = F.layer_norm(P, (d,), f["ln_kv_gamma"], f["ln_kv_beta"], w["ln_eps"])
        at = offs[a:b, None] - offs[a] + np.minimum(np.arange(4)[None], n[a:b, None] - 1)
        P = P[torch.from_numpy(at).long().to(dev)].view(b - a, 4, h, d // h)
        scores = (P * f["query"]).sum(-1) / math.sqrt(d // h)
        there = torch.from_numpy(np.arange(4)[None] < n[a:b, None]).to(dev)
        alpha = scores.masked_fill(~there[..., None], -math.inf).softmax(1)
        o = (alpha[..., None] * P).sum(1).reshape(b - a, d)
        out[a:b] = F.layer_norm(F.gelu(o @ f["w_o"].T + f["b_o"]), (d,), f["ln_o_gamma"], f["ln_o_beta"], w["ln_eps"])
    return out


def _attend64(q, K, V):
    """q [Hq][D], K and V [n][Hkv][D]."""
    hkv, D = K.shape[1:]
    q = q.double().view(hkv, -1, D)
    return ((q @ K.permute(1, 2, 0)) / math.sqrt(D)).softmax(-1).matmul(V.transpose(0, 1)).reshape(-1, D)


def _entries64(x, layer, b, n):
    """K and V [n][Hkv][D] of the first n entries of sequence b."""
    t = torch.arange(n, device=x["pool"].device)
    pages = torch.from_numpy(x["table"][b]).to(t.device).long()[t // PAGE]
    e = x["pool"][layer][pages, :, :, t % PAGE].double()
    return e[:, 0], e[:, 1]


def _rollback64(x, case):
    """[(K, V)] of every sequence after the rollback, and each kept entry's shift."""
    so, ss, sn = x["spans"]
    got = []
    for b, L in enumerate(x["lens"]):
        K, V = _entries64(x, 0, b, int(L))
        s, n = ss[so[b]:so[b + 1]], sn[so[b]:so[b + 1]]
        src = np.zeros(int(L), np.int64)          # 1: starts a span, -1: dropped
        for i in range(1, 4):
            src[(s + i)[n > i]] = -1
        src[s] = 1
        kept = np.nonzero(src >= 0)[0]
        shift = torch.from_numpy(np.where(src[kept] == 1, 0, kept - np.arange(len(kept)))).to(K.device)
        to = torch.from_numpy(np.nonzero(src[kept] == 1)[0]).to(K.device)
        kept = torch.from_numpy(kept).to(K.device)
        K, V = K[kept], V[kept]
        if "freq" in x:
            half = case["D"] // 2
            a = (shift[:, None] * x["freq"].double())[:, None]
            c, sine, u, v = a.cos(), a.sin(), K[..., :half], K[..., half:]
            K = torch.cat([u * c + v * sine, v * c - u * sine], -1)
        K[to], V[to] = x["sk"][so[b]:so[b + 1], 0].double(), x["sv"][so[b]:so[b + 1], 0].double()
        got.append((K, V))
    return got


def exact(case, seed):
    x, r = _inputs(case, seed)
    kind, out = case["kind"], []
    if kind == "rules":
        return None                               # copies and whole numbers
    if kind in ("step", "merge", "prompt"):
        z = _merge64(x, case)
        out.append(z)
    if kind in ("step", "context"):
        kv = _rollback64(x, case)
        out.append(torch.stack([_attend64(x["q"][0, b], K, V) for b, (K, V) in enumerate(kv)]))
        out += [None, None, None]
        pool = None
        if "freq" in x:                           # re-rotated keys are computed numbers
            pool = x["pool"].double()
            for b, (K, V) in enumerate(kv):
                t = torch.arange(int(x["spans"][1][x["spans"][0][b]]), len(K), device=K.device)
                pages = torch.from_numpy(x["table"][b]).to(t.device).long()[t // PAGE]
                pool[0][pages, :, :, t % PAGE] = torch.stack([K[t], V[t]], 1)
        out.append(pool)
    if kind in ("layers", "engine"):
        o = torch.empty_like(x["q"], dtype=torch.float64)
        for l in range(case["layers"]):
            for b, L in enumerate(x["lens"]):
                k, row = int(x["merge_k"][b]), int(x["merge_row"][b])
                K, V = _entries64(x, l, b, int(L) + 1 - k if k else int(L))
                new = (x["sk"][row, l], x["sv"][row, l]) if k else (x["nk"][b, l], x["nv"][b, l])
                K, V = (torch.cat([t, n.double()[None]]) for t, n in zip((K, V), new))
                o[l, b] = _attend64(x["q"][l, b], K, V)
        out += [o, None, None, None, None]
    if kind == "prompt":
        so, ss, sn = x["spans"]
        embeds = torch.zeros((case["B"] * case["L"], case["d"]), dtype=torch.float64, device=z.device)
        rows = []
        for b in range(case["B"]):
            src = x["tokens"][b].astype(np.int64)
            for i in range(1, 4):
                src[(ss + i)[so[b]:so[b + 1]][sn[so[b]:so[b + 1]] > i]] = -1 << 40
            src[ss[so[b]:so[b + 1]]] = -1 - np.arange(so[b], so[b + 1])
            rows.append(src[src > -1 << 39])
        rows = torch.from_numpy(np.concatenate(rows)).to(z.device)
        embeds[:len(rows)] = x["emb"][rows.clamp(min=0)].double()
        at = torch.nonzero(rows < 0)[:, 0]
        embeds[at] = z[-1 - rows[at]]
        out += [embeds, None, None]
    if kind == "prefill":
        o = torch.empty(x["q"].shape, dtype=torch.float64, device=x["q"].device)
        G = case["hq"] // case["hkv"]
        for a, b in zip(x["cu"][:-1], x["cu"][1:]):
            n = int(b - a)
            mask = torch.ones((n, n), dtype=torch.bool, device=o.device).triu(1)
            for g in range(case["hkv"]):
                q = x["q"][a:b, g * G:(g + 1) * G].double().transpose(0, 1)
                p = (q @ x["k"][a:b, g].double().T / math.sqrt(case["D"])).masked_fill(mask, -math.inf).softmax(-1)
                o[a:b, g * G:(g + 1) * G] = (p @ x["v"][a:b, g].double()).transpose(0, 1)
        out.append(o)
    if kind == "distill":
        so, ss, sn = x["spans"]
        V, t_rows, s_rows, t0, s0 = case["V"], [], [], 0, 0
        for b, L in enumerate(x["lens"]):
            s, n = ss[so[b]:so[b + 1]], sn[so[b]:so[b + 1]]
            keep = np.ones(int(L), bool)
            for i in range(0, 3):
                keep[(s + i)[n > i + 1]] = False   # a span keeps its last position
            first = int(s[0]) if len(s) else int(L)
            kept = np.nonzero(keep)[0]
            pos = np.arange(len(kept))
            t_rows.append(t0 + kept[kept >= first])
            s_rows.append(s0 + pos[kept >= first])
            t0, s0 = t0 + int(L), s0 + len(kept)
        t_rows, s_rows = (torch.from_numpy(np.concatenate(a)).to(x["student"].device) for a in (t_rows, s_rows))
        N = len(t_rows)
        pair = torch.zeros(x["student"].shape[0], dtype=torch.float64, device=t_rows.device)
        grad = torch.zeros(x["student"].shape, dtype=torch.float64, device=t_rows.device) if case["grad"] else None
        for i in range(0, N, 512):
            T = x["teacher"][t_rows[i:i + 512], :V].double().softmax(-1)
            P = x["student"][s_rows[i:i + 512], :V].double().softmax(-1)
            lg = (P + case["eps"]).log()
            pair[i:i + len(T)] = -(T * lg).sum(-1)
            if grad is not None:
                a = T * P / (P + case["eps"])
                grad[s_rows[i:i + 512], :V] = (P * a.sum(-1, keepdim=True) - a) / N
        out += [pair.sum().view(1) / max(N, 1), pair, None, None, None, None]
        out += [grad] if case["grad"] else []
    return out + [None]
