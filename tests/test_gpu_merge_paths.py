"""How the merge module lays out its products, seen in its workspace (every CTA of GEMM1, the pooling, the W_o
conversion and GEMM2 writes a word of its own on every call), and each layout against the float64 oracle (the tolerance
of every merge test).  Sizes follow the GPU's SM count, so that no case drifts to another layout."""
import pytest
import torch

import oracle
from oracle import merge as M
import workloads as W
from helpers import dev, float_close, umim
from test_gpu_merge import _weights_with

pytestmark = pytest.mark.gpu

KERNELS, CTAS = 4, 1024   # words at the end of the workspace: one per kernel and CTA


def run(case):
    """(z, status, {kernel: CTAs that ran})."""
    m, on = umim(), dev()
    d, S, T = case.weights.d_model, case.span_offsets.numel() - 1, case.token_ids.numel()
    ws = torch.full((m.umim_merge_spans_workspace_size(T, S, d),), 0x7F, dtype=torch.uint8, device=on)
    status = m.new_status(on)
    z = m.umim_merge_spans(case.table.to(on), case.token_ids.to(on), case.span_offsets.to(on), case.weights.to(on),
                           surrogates=torch.full((S, d), 12345.0, device=on), workspace_buf=ws, dev_status=status)
    torch.cuda.synchronize()
    words = ws[-KERNELS * CTAS * 4:].view(torch.int32).view(KERNELS, CTAS).cpu()
    ran = [int((w != 0x7F7F7F7F).sum()) for w in words]
    return z, int(status.item()), dict(zip(("gemm1", "pool", "w_o", "gemm2"), ran))


def sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


def tiles(rows, d):
    return -(-rows // 128) * (d // 256)


def check(case):
    z, status, ran = run(case)
    assert status == 0
    wf = M.weights_f64({n: W.bits(v) for n, v in case.weights.tensors().items()})
    float_close(z.cpu().double().numpy(),
                oracle.merge_spans(W.bits(case.table), case.token_ids.numpy(), case.span_offsets.numpy(), wf,
                                   case.weights.n_heads))
    return ran


# a cluster of eight takes its SMs from one GPC: a tenth of the SMs' number of them fit at once (15 of 152 SMs), and
# the next number of tiles is split in four
@pytest.mark.parametrize("d", [512, 2048])
@pytest.mark.parametrize("more", [0, 1])
def test_clusters_of_eight_fit_at_once(d, more):
    rows = (sms() // 10) // (d // 256) + more   # row tiles
    case = W.merge_case(770 + d + more, vocab=500, d=d, h=4, n_spans=rows * 128 - 27, kmin=1, kmax=1)
    ran = check(case)
    for g in ("gemm1", "gemm2"):
        assert ran[g] == tiles(rows * 128, d) * (4 if more else 8)


# GEMM1 unsplit with room for the W_o conversion in its side warp: GEMM2 is split in four or not at all, never in two
@pytest.mark.parametrize("d,tiles2,split2", [(512, 0.2, 4), (512, 0.24, 1), (512, 0.4, 1), (1024, 0.24, 1)])
def test_output_projection_is_not_split_in_two_beside_a_side_warp(d, tiles2, split2):
    rows = int(sms() * tiles2) // (d // 256)
    case = W.merge_case(780 + rows, vocab=500, d=d, h=4, n_spans=rows * 128 - 5, kmin=4, kmax=4)
    ran = check(case)
    t1 = tiles(case.token_ids.numel(), d)
    assert ran["gemm1"] == min(t1, sms())
    assert ran["gemm2"] == tiles(rows * 128, d) * split2
    assert ran["w_o"] == 0   # no conversion kernel: in the split product or in GEMM1's side warp


def split_of(rows, d):
    """The rule: as many CTAs a tile as keep every cluster resident (4/5 of the SMs for clusters of eight, else 7/8)."""
    n = sms()
    for s in (8, 4, 2):
        if tiles(rows, d) * s <= (n // 5 * 4 if s == 8 else n // 8 * 7) and d // 64 % s == 0:
            return s
    return 1


def layout(S, T, d):
    """(CTAs of GEMM1, of GEMM2, whether W_o has a kernel of its own, GEMM1's split, GEMM2's split)."""
    s1, s2 = split_of(T, d), split_of(S, d)
    whole = min(tiles(T, d), sms())
    side_warp = s1 == 1 and d * d // 8 <= 128 * 32 * whole * (tiles(T, d) // whole)
    if s2 == 2 and side_warp:
        s2 = 1
    ctas = lambda rows, s: tiles(rows, d) * s if s > 1 else min(tiles(rows, d), sms())
    return ctas(T, s1), ctas(S, s2), s2 == 1 and not side_warp, s1, s2


# on 152 SMs: every split of both products; three, two and one K steps a CTA (fewer than the ring's stages); the widest
LAYOUTS = [(512, 9, 1), (512, 300, 4), (512, 700, 4), (512, 1200, 4), (512, 2100, 2), (512, 4300, 1), (1024, 450, 4),
           (1536, 40, 2), (1536, 240, 2), (2048, 200, 1), (2048, 1100, 1), (8192, 3, 2), (8192, 150, 1)]


def test_layouts_hold_every_split():
    got = [layout(S, S * k, d)[2:] for d, S, k in LAYOUTS]
    assert {1, 2, 4, 8} == {g[1] for g in got} == {g[2] for g in got}
    assert True in {g[0] for g in got}   # W_o's own kernel


@pytest.mark.parametrize("d,S,k", LAYOUTS)
def test_layouts_match_oracle(d, S, k):
    case = W.merge_case(790 + S, vocab=400, d=d, h=8, n_spans=S, kmin=k, kmax=k)
    ran = check(case)
    g1, g2, conversion, _, _ = layout(S, S * k, d)
    assert (ran["gemm1"], ran["gemm2"], ran["w_o"] > 0) == (g1, g2, conversion)


# the three places where W_o becomes fp16: inside the split product, GEMM1's side warp, a kernel of its own
def _place(name):
    d, S = {"split": (512, 9), "side_warp": (512, 128 * (sms() // 8 * 7 // 4 + 1) - 3),
            "kernel": (2048, 128 * (sms() // 8 * 7 // 16 + 1) - 5)}[name]
    _, _, conversion, _, s2 = layout(S, S, d)
    assert (s2 > 1, conversion) == {"split": (True, False), "side_warp": (False, False), "kernel": (False, True)}[name]
    return W.merge_case(800 + d + S, vocab=300, d=d, h=4, n_spans=S, kmin=1, kmax=1)


@pytest.mark.parametrize("place", ["split", "side_warp", "kernel"])
@pytest.mark.parametrize("what", ["b_kv", "embedding", "w_o", "b_o"])
def test_values_past_fp16_are_refused(place, what):
    """In the first product's output (a bias, a token's row), in W_o times 256, in the second product's output; the
    value concerns one column or token."""
    case = _place(place)
    table, weights = case.table, case.weights
    if what == "embedding":
        table = table.clone()
        table[case.token_ids[-1]] = 3.0e6
    else:
        t = getattr(weights, what).clone()
        if what == "w_o":
            t[-3, 5] = 300.0
        else:
            t[-7] = 70000.0
        weights = _weights_with(case, **{what: t})
    z, status, _ = run(W.MergeCase(table=table, token_ids=case.token_ids, span_offsets=case.span_offsets, weights=weights))
    assert status == 2   # UMIM_ERR_UNSUPPORTED
    assert torch.all(z == 12345.0)   # nothing written


@pytest.mark.parametrize("place", ["split", "side_warp", "kernel"])
def test_tiny_output_weights_keep_their_precision(place):
    """Entries that would be fp16 subnormals without the power-of-two staging."""
    case = _place(place)
    small = {n: (getattr(case.weights, n).float() * 1e-6).to(torch.bfloat16) for n in ("w_o", "b_o")}
    check(W.MergeCase(table=case.table, token_ids=case.token_ids, span_offsets=case.span_offsets,
                      weights=_weights_with(case, **small)))
