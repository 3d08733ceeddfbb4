"""Launches too small to fill the GPU: their prompt spans are shared out
evenly over several splits, whose states the merge kernel takes up to sixteen
of at a time (spans of 512 keys per split at the least; up to eight splits, in
delta mode four plus four of delta rows; up to eight generated-span splits).

Outputs against the oracle at the edges of the splits, the same bits in every
pass order, and the same bits for cells that read the clean span whether the
other cells of the batch are patched or not."""
import numpy as np
import pytest
import torch

import oracle
from paper_2605_30574_gb300 import build as B
from paper_2605_30574_gb300 import splice as S
from paper_2605_30574_gb300.sweep import SweepBatch
from paper_2605_30574_gb300.synth import workloads as WL
from parity_util import CachedInputs, assert_close

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    B.build()


def workload(Tp, d, hq, hkv, P, T, window=0):
    return WL.Workload(f"small-{Tp}-{d}-{P}", 2, hq, hkv, d, P, Tp, (WL.SAME_ALGO, WL.ZERO, WL.BLANK), T, (0, 1, 2),
                       (0, 3), 8, 4, batch=10 ** 6, sliding_window=window, global_every=0)


# the smallest span with two splits and one key less; one key into a block; a
# span of eight splits and one of more than eight times the least
@pytest.mark.parametrize("Tp", [1023, 1024, 1025, 1537, 2049, 4097, 5000])
@pytest.mark.parametrize("d,hq,hkv,P", [(64, 2, 1, 1), (128, 12, 4, 2), (256, 4, 2, 1)])
def test_span_splits(Tp, d, hq, hkv, P):
    t = 70
    wl = workload(Tp, d, hq, hkv, P, t)
    seqs = wl.sequences()
    a = SweepBatch(wl, seqs=seqs)
    b = SweepBatch(wl, seqs=[WL.Seq(q.prompt, q.slot, wl.num_layers, q.W) for q in seqs])
    inp = CachedInputs(wl)
    for l, step in ((0, 2), (1, t)):
        a.gen_inputs(l, step)
        outs = []
        for order in (0, 1, 2):
            S.splice_debug_pass_order(a.desc, order)
            a.out.fill_(float("nan"))
            a.step(l, step)
            outs.append(a.out.clone())
        S.splice_debug_pass_order(a.desc, 0)
        assert torch.equal(outs[0], outs[1]) and torch.equal(outs[0], outs[2]), (l, step)
        m = S.splice_debug_source_map(a.desc, l, step)
        clean = [s for s in range(a.B) if m[s] == S.SRC_CLEAN]
        assert clean
        assert torch.equal(b.run(l, step)[clean], outs[0][clean]), (l, step)
        which = sorted({0, a.B // 2, a.B - 1, clean[0]})
        ref = np.stack([oracle.decode_attn(wl, inp, s, seqs[s], l, step) for s in which])
        assert_close(outs[0][which].cpu().numpy(), ref, f"Tp={Tp} d={d} l={l} t={step}")
    S.splice_check_device_error(a.desc)
    S.splice_check_device_error(b.desc)


@pytest.mark.parametrize("d,hq,hkv", [(64, 2, 1), (128, 4, 2), (256, 2, 1)])
@pytest.mark.parametrize("Tp,t", [(2100, 600), (4100, 33), (4500, 513)])
def test_many_partials_and_delta_rows(Tp, t, d, hq, hkv):
    """Up to eight span splits with eight generated-span splits, and in delta
    mode four span splits, four of delta rows and eight generated ones."""
    wl = workload(Tp, d, hq, hkv, 1, t)
    seqs = wl.sequences()
    a = SweepBatch(wl, seqs=seqs)
    inp = CachedInputs(wl)
    which = list(range(0, a.B, 3))
    ref = np.stack([oracle.decode_attn(wl, inp, s, seqs[s], 1, t) for s in which])
    assert_close(a.run(1, t)[which].cpu().numpy(), ref, f"Tp={Tp} d={d}")
    buf = torch.empty(S.splice_delta_bytes(a.desc), dtype=torch.uint8, device="cuda")
    S.splice_delta_build(a.desc, a.k_clean, a.v_clean, a.k_donor, a.v_donor, buf)
    assert_close(a.run(1, t)[which].cpu().numpy(), ref, f"delta Tp={Tp} d={d}")
    S.splice_check_device_error(a.desc)


def test_windows_shorter_than_the_span():
    """The visible part of the span, and with it the splits, moves with the step."""
    wl = workload(3000, 128, 8, 2, 1, 900, window=1500)
    seqs = wl.sequences()
    a = SweepBatch(wl, seqs=seqs)
    inp = CachedInputs(wl)
    for step in (1, 470, 480, 900):
        which = [0, a.B - 1]
        ref = np.stack([oracle.decode_attn(wl, inp, s, seqs[s], 1, step) for s in which])
        assert_close(a.run(1, step)[which].cpu().numpy(), ref, f"t={step}")
    S.splice_check_device_error(a.desc)


# eight and three rows on the tensor-core kernel, one on the FMA kernel; a step
# whose generated spans are short beside the prompts' and the first whole block
@pytest.mark.parametrize("d,hq,hkv,cells", [(256, 16, 2, 420), (128, 12, 4, 500), (64, 4, 4, 1400)])
def test_short_generated_spans_beside_long_prompts(d, hq, hkv, cells):
    """The prompt-span pass goes first, and the merge kernel merges (three
    launches and the same bits as with the passes the other way round)."""
    wl = workload(2100, d, hq, hkv, 4, 16)
    seqs = (wl.sequences() * (cells // len(wl.sequences()) + 1))[:cells]
    b = SweepBatch(wl, seqs=seqs)
    inp = CachedInputs(wl)
    for l, t in ((0, 3), (1, 16)):
        b.gen_inputs(l, t)
        outs = []
        for order in (1, 2):
            S.splice_debug_pass_order(b.desc, order)
            b.out.fill_(float("nan"))
            before = S.splice_kernel_launches(b.desc)
            b.step(l, t)
            torch.cuda.synchronize()
            assert S.splice_kernel_launches(b.desc) - before == 3
            outs.append(b.out.clone())
        S.splice_debug_pass_order(b.desc, 0)
        assert torch.equal(*outs), (l, t)
        which = [0, cells // 2, cells - 1]
        ref = np.stack([oracle.decode_attn(wl, inp, s, seqs[s], l, t) for s in which])
        assert_close(outs[0][which].cpu().numpy(), ref, f"d={d} l={l} t={t}")
    S.splice_check_device_error(b.desc)
