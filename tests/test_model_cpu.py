"""Host-side pieces of the end-to-end decoder (Algorithm 1), on the CPU.

* donor token sequences follow Table 1's structure: the scaffold is kept,
  BLANK fills the content with one filler token, SAME_ALGO / DIFF_ALGO
  replace the ladder's fractions (0.1 / 0.5) of content positions, ZERO has
  no tokens;
* RoPE preserves norms and makes q . k depend only on the position offset;
* prefill is causal: a position's K and V do not depend on later tokens.
"""
import math

import pytest
import torch

from paper_2605_30574_gb300 import decoder as K
from paper_2605_30574_gb300.model import DecoderDims, RandomDecoder, _own, donor_tokens, tiny_dims
from paper_2605_30574_gb300.synth import workloads as W


@pytest.fixture(scope="module")
def model():
    return RandomDecoder(tiny_dims(), seed=0, device="cpu")


def test_donor_tokens_follow_table1():
    g = torch.Generator()
    g.manual_seed(3)
    vocab, Tp, head, tail, filler = 50000, 4096, 24, 12, 7
    prompt = torch.randint(0, vocab, (Tp,), generator=g)
    content = slice(head, Tp - tail)
    n = Tp - head - tail
    assert donor_tokens(prompt, W.ZERO, g, vocab, head, tail, filler) is None
    for kind in (W.BLANK, W.SAME_ALGO, W.DIFF_ALGO, W.DIFF_FAMILY):
        d = donor_tokens(prompt, kind, g, vocab, head, tail, filler)
        assert d.shape == prompt.shape
        assert torch.equal(d[:head], prompt[:head]) and torch.equal(d[Tp - tail:], prompt[Tp - tail:])
    blank = donor_tokens(prompt, W.BLANK, g, vocab, head, tail, filler)
    assert bool((blank[content] == filler).all())
    for kind, p in ((W.SAME_ALGO, 0.1), (W.DIFF_ALGO, 0.5)):
        d = donor_tokens(prompt, kind, g, vocab, head, tail, filler)
        changed = int((d[content] != prompt[content]).sum())
        # binomial(n, p) within 5 standard deviations (a replaced token equals
        # the old one with probability 1 / vocab)
        assert abs(changed - n * p) < 5 * math.sqrt(n * p * (1 - p)) + 2, (kind, changed)
    fam = donor_tokens(prompt, W.DIFF_FAMILY, g, vocab, head, tail, filler)
    assert int((fam[content] != prompt[content]).sum()) > n - 10


def test_rope_is_a_relative_rotation(model):
    g = torch.Generator()
    g.manual_seed(1)
    d = model.dims.head_dim
    q = torch.randn(1, 1, d, generator=g)
    k = torch.randn(1, 1, d, generator=g)
    for m, n, c in ((5, 2, 100), (0, 31, 7), (400, 3, 1000)):
        qm, kn = model.rope(q, torch.tensor([m])), model.rope(k, torch.tensor([n]))
        assert torch.allclose(qm.norm(), q.norm(), rtol=1e-5)
        a = (qm * kn).sum()
        b = (model.rope(q, torch.tensor([m + c])) * model.rope(k, torch.tensor([n + c]))).sum()
        assert torch.allclose(a, b, rtol=1e-4, atol=1e-4), (m, n, c)


def test_prefill_is_causal(model):
    dims = model.dims
    g = torch.Generator()
    g.manual_seed(2)
    Tp = 24
    toks = torch.randint(0, dims.vocab, (Tp,), generator=g)
    alt = toks.clone()
    alt[-1] = (alt[-1] + 1) % dims.vocab
    shape = (dims.num_layers, dims.num_kv_heads, Tp, dims.head_dim)
    k1, v1, k2, v2 = (torch.empty(shape, dtype=torch.bfloat16) for _ in range(4))
    l1 = model.prefill(toks, k1, v1)
    l2 = model.prefill(alt, k2, v2)
    assert torch.equal(k1[:, :, :-1], k2[:, :, :-1]) and torch.equal(v1[:, :, :-1], v2[:, :, :-1])
    assert not torch.equal(k1[:, :, -1], k2[:, :, -1])
    assert not torch.equal(l1, l2)


# An MLP of another input width has no kernels: the torch expressions refuse it.
@pytest.mark.parametrize("gate,up,down", [((512, 128), (512, 128), (128, 512)), ((512, 320), (512, 320), (320, 512)),
                                          ((512, 256), (512, 128), (256, 512)), ((512, 256), (512, 256), (128, 512))])
def test_kernels_take_only_an_mlp_of_the_models_width(model, monkeypatch, gate, up, down):
    monkeypatch.setattr(K, "plain", lambda acts, weights: True)
    h = torch.zeros(3, model.dims.d_model)
    assert model._kernels(0, h)
    kept = dict(model.layers[0])
    for n, shape in (("w_gate", gate), ("w_up", up), ("w_down", down)):
        monkeypatch.setitem(model.layers[0], n, torch.zeros(shape, dtype=torch.bfloat16))
    assert not model._kernels(0, h)
    monkeypatch.undo()
    assert all(model.layers[0][n] is kept[n] for n in kept)


# The kernel reads the head norms' weights in words of d / 64 elements: views
# that do not start on one (of a flat buffer of all parameters, say) are torch's.
@pytest.mark.parametrize("d", [64, 128, 256])
@pytest.mark.parametrize("name", ["q_norm", "k_norm"])
def test_kernels_take_only_head_norms_on_whole_words(monkeypatch, d, name):
    monkeypatch.setattr(K, "plain", lambda acts, weights: True)
    model = RandomDecoder(DecoderDims(1, 2, 1, d, 64, 64, 8), device="cpu")
    h, pos = torch.zeros(3, 64), torch.arange(3)
    flat = torch.ones(d + 8, dtype=torch.bfloat16)
    for at in range(8):
        model.layers[0][name] = flat[at:at + d]
        assert model._kernels(0, h, pos) == (at % (d // 64) == 0)


def test_a_piece_of_ones_own_is_the_one_that_runs(monkeypatch):
    """A decoder that brings its own rope or qkv -- by a subclass, on an
    instance, or patched into the class -- is not passed by."""
    calls = []

    class Unturned(RandomDecoder):
        def rope(self, x, pos):
            calls.append("rope")
            return x

    class Spy(RandomDecoder):
        def qkv(self, l, h, pos):
            calls.append("qkv")
            return super().qkv(l, h, pos)

    dims = DecoderDims(1, 2, 1, 64, 64, 64, 8)
    tokens, h, pos = torch.arange(5), torch.zeros(5, 64), torch.arange(5)
    stores = [torch.zeros(1, 1, 5, 64, dtype=torch.bfloat16) for _ in range(2)]
    plain, a, b, c = (cls(dims, device="cpu") for cls in (RandomDecoder, Unturned, RandomDecoder, Spy))
    b.rope = lambda x, pos: calls.append("rope") or x
    for m in (a, b):
        m.qkv(0, h, pos)
        m.prefill(tokens, *stores)
    c.prefill(tokens, *stores)
    assert calls == ["rope"] * 8 + ["qkv"]
    monkeypatch.setattr(K, "plain", lambda acts, weights: True)
    assert plain._kernels(0, h, pos) and c._kernels(0, h, pos)
    assert not a._kernels(0, h, pos) and not b._kernels(0, h, pos)
    assert _own(plain, "qkv") and _own(a, "qkv") and not _own(c, "qkv")
    b.qkv = b.qkv
    assert _own(b, "qkv")
    b.qkv = lambda l, h, pos: None
    assert not _own(b, "qkv")
    monkeypatch.setattr(RandomDecoder, "rope", Unturned.rope)
    assert not plain._kernels(0, h, pos)


class Scaled(RandomDecoder):
    """Its own block_out, which reads the attention output as fp32."""

    def block_out(self, l, h, attn):
        assert attn.dtype is torch.float32
        return super().block_out(l, h, attn * torch.ones((), dtype=torch.float32))


def test_a_block_out_of_ones_own_gets_the_attention_in_fp32():
    dims = DecoderDims(1, 2, 1, 64, 64, 64, 8)
    stores = [torch.zeros(1, 1, 5, 64, dtype=torch.bfloat16) for _ in range(2)]
    got = Scaled(dims, device="cpu").prefill(torch.arange(5), *stores)
    assert torch.equal(got, RandomDecoder(dims, device="cpu").prefill(torch.arange(5), *stores))


# (other lengths, head dims and head counts than the queries'; unlike shapes)
@pytest.mark.parametrize("k,v", [((2, 5, 64), (2, 5, 64)), ((2, 7, 64), (2, 7, 64)), ((2, 6, 128), (2, 6, 128)),
                                 ((3, 6, 64), (3, 6, 64)), ((2, 6, 64), (2, 5, 64)), ((2, 6, 64), (1, 6, 64)),
                                 ((2, 6, 64), (2, 6, 128))])
def test_prefill_attention_kernel_takes_matching_keys_only(k, v):
    """A qkv of one's own may return others, which torch's attention refuses."""
    q, k, v = (torch.zeros(s, dtype=torch.bfloat16) for s in ((6, 4, 64), k, v))
    assert K.causal(q, k, v, 0.125) is None
