"""How the merge module lays out its products, seen in its workspace (every CTA of GEMM1, the pooling, the W_o
conversion and GEMM2 writes a word of its own on every call), and each layout against the float64 oracle (the tolerance
of every merge test).  Sizes follow the GPU's SM count, so that no case drifts to another layout."""
import pytest
import torch

import oracle
from oracle import merge as M
import workloads as W
from helpers import dev, float_close, umim

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
