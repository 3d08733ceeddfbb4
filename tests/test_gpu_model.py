"""Algorithm 1 end to end with a random-initialised decoder.

The library's decode (prefill into the clean and donor stores, then per step
and layer ``suffix_kv_append`` + ``spliced_decode_attn``) is compared with the
same decoder whose decode attention is the fp64 oracle over a physically
spliced copy of each sequence's cache: at step t every patched layer
(l >= L, t >= W) reads the donor span (or zeros for ZERO) in place of the
prompt span, as Algorithm 1's in-place replacement leaves it.  Teacher
forcing: both paths take the library's own greedy tokens as inputs, so the
per-step logits are compared at every step; each path keeps the generated
K/V of its own earlier forward passes.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2605_30574_gb300 import build as B
from paper_2605_30574_gb300 import decoder as K
from paper_2605_30574_gb300.model import RandomDecoder, SpliceDecode, tiny_dims
from paper_2605_30574_gb300.synth import workloads as WL

pytestmark = pytest.mark.gpu

# Tolerance on logits, relative to the step's largest |logit|: the attention
# output differs from the fp64 oracle by up to ~1e-3 (bf16 probabilities in
# the prompt-span pass; the attention tests' bound is 1e-2), and the
# decoder's bf16 projections of that output round at 2^-9 relative.
LOGIT_TOL = 2e-2


@pytest.fixture(scope="module", autouse=True)
def _built():
    B.build()


def reference_step(run: SpliceDecode, t: int, tokens: torch.Tensor, ref_k: np.ndarray, ref_v: np.ndarray):
    """Logits of step t with oracle attention; ref_k/ref_v [B][N][Hkv][T][d]
    hold this path's own generated K/V (entry t-1 is written here)."""
    model, dims = run.model, run.model.dims
    pos = torch.full((run.B,), run.Tp + t - 1, device=model.device)
    h = model.embed[tokens].float()
    kc = run.k_clean.double().cpu().numpy()
    vc = run.v_clean.double().cpu().numpy()
    kd = run.k_donor.double().cpu().numpy() if run.k_donor is not None else None
    vd = run.v_donor.double().cpu().numpy() if run.v_donor is not None else None
    for l in range(dims.num_layers):
        q, k, v = model.qkv(l, h, pos)
        ref_k[:, l, :, t - 1] = k.double().cpu().numpy()
        ref_v[:, l, :, t - 1] = v.double().cpu().numpy()
        qn = q.double().cpu().numpy()
        attn = np.zeros(qn.shape, np.float64)
        for s, cell in enumerate(run.seqs):
            kind = run.slot_kinds[cell.slot]
            src = oracle.splice_source(cell.L, cell.W, cell.slot, kind, l, t)
            if src == oracle.SRC_CLEAN:
                pk, pv = kc[cell.prompt, l], vc[cell.prompt, l]
            elif src == oracle.SRC_ZERO:
                pk, pv = np.zeros_like(kc[cell.prompt, l]), np.zeros_like(vc[cell.prompt, l])
            else:
                i = run.stored.index(src - oracle.SRC_DONOR0)
                pk, pv = kd[cell.prompt, i, l], vd[cell.prompt, i, l]
            K = np.concatenate([pk, ref_k[s, l, :, :t]], axis=1)
            V = np.concatenate([pv, ref_v[s, l, :, :t]], axis=1)
            attn[s] = oracle.attend(qn[s], K, V, 0, model.sm_scale)
        h = model.block_out(l, h, torch.from_numpy(attn).to(model.device, torch.float32))
    return model.logits(h)


def test_algorithm1_teacher_forced_matches_oracle_attention():
    dims = tiny_dims()
    model = RandomDecoder(dims, seed=0)
    P, Tp, T = 2, 48, 8
    gen = torch.Generator(device="cuda")
    gen.manual_seed(11)
    prompts = torch.randint(0, dims.vocab, (P, Tp), generator=gen, device="cuda")
    kinds = (WL.BLANK, WL.ZERO, WL.SAME_ALGO)
    seqs = [WL.Seq(p, k, L, Wv) for p in range(P) for k in range(len(kinds)) for L in (0, 2, dims.num_layers)
            for Wv in (0, 2, 5)]
    run = SpliceDecode(model, prompts, kinds, seqs, T, scaffold_head=4, scaffold_tail=2, filler=3)
    toks = run.decode(T)
    # y_0 comes from the clean prefill
    assert torch.equal(toks[:, 0], run.first_token)
    ref_k = np.zeros((run.B, dims.num_layers, dims.num_kv_heads, T, dims.head_dim))
    ref_v = np.zeros_like(ref_k)
    worst = 0.0
    for t in range(1, T):
        ours = run.step(t, toks[:, t - 1])
        # the library path reproduces its own greedy choice
        assert torch.equal(ours.argmax(-1), toks[:, t]), t
        ref = reference_step(run, t, toks[:, t - 1], ref_k, ref_v)
        scale = ref.abs().max().item()
        err = (ours - ref).abs().max().item() / scale
        worst = max(worst, err)
        assert err < LOGIT_TOL, (t, err)
        # where the reference's choice is clear, it is the same token
        top2 = ref.topk(2, dim=-1).values
        clear = (top2[:, 0] - top2[:, 1]) > 2 * LOGIT_TOL * scale
        assert torch.equal(ref.argmax(-1)[clear], toks[clear, t]), t
    print(f"worst relative logit error {worst:.2e}")
    run.close()


def test_splice_changes_patched_cells_only():
    """Cells with L = N (no layer patched) decode exactly like the clean-only
    decode of the same prompt; ZERO cells patched from step 1 at every layer
    generate from a different cache and differ in logits."""
    dims = tiny_dims()
    model = RandomDecoder(dims, seed=1)
    P, Tp, T = 1, 40, 6
    gen = torch.Generator(device="cuda")
    gen.manual_seed(5)
    prompts = torch.randint(0, dims.vocab, (P, Tp), generator=gen, device="cuda")
    kinds = (WL.ZERO, WL.BLANK)
    N = dims.num_layers
    seqs = [WL.Seq(0, 0, N, 0), WL.Seq(0, 1, N, 0), WL.Seq(0, 0, 0, 0), WL.Seq(0, 1, 0, 1)]
    run = SpliceDecode(model, prompts, kinds, seqs, T, scaffold_head=2, scaffold_tail=2, filler=3)
    toks = run.decode(T)
    # the two never-patched cells are the same decode
    assert torch.equal(toks[0], toks[1])
    # patched cells see another prompt span from step 1 on
    l0 = run.step(1, toks[:, 0])
    assert not torch.equal(l0[2], l0[0]) and not torch.equal(l0[3], l0[0])
    run.close()


def test_a_wait_that_ran_out_in_the_prefills_is_reported(monkeypatch):
    """A prefill's outputs are then wrong; the prefills' end says so (the
    library's own call, but for the word that it reads)."""
    real, reads = K.lib(), []

    class Library:
        def __getattr__(self, name):
            return getattr(real, name)

        def decoder_error(self, ref):
            rc = real.decoder_error(ref)
            reads.append(1)
            if len(reads) > 1:                  # (the first is the reader's making)
                ref._obj.value = 0x10
            return rc

    monkeypatch.setattr(K, "_LIB", Library())
    monkeypatch.setattr(K, "_records", {})
    model = RandomDecoder(tiny_dims(), seed=0)
    prompts = torch.randint(0, model.dims.vocab, (1, 20), device="cuda")
    with pytest.raises(RuntimeError, match="0x10"):
        SpliceDecode(model, prompts, (WL.SAME_ALGO, WL.ZERO), [WL.Seq(0, 0, 0, 0)], 4, 2, 2, filler=3)
