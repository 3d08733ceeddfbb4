"""The decoder's kernels against the torch expressions they stand in for.

Both compute in fp32 with the same element operations and round to bf16 at the
same places; only the order of a row's sum differs.  A sum of D squares in
another order moves rms by at most about D 2^-24 relative, far below the
spacing of bf16, so a bf16 output differs by one unit in the last place at
most (2^-7 relative, at a rounding boundary) -- after RoPE, by one unit of the
larger of the two rotated terms.
"""
import pytest
import torch

from paper_2605_30574_gb300 import build as B
from paper_2605_30574_gb300 import decoder as K
from paper_2605_30574_gb300.model import DecoderDims, RandomDecoder, _rms_norm

pytestmark = pytest.mark.gpu
ULP = 2.0 ** -7


@pytest.fixture(scope="module", autouse=True)
def _built():
    B.build()


def gen(seed=0):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def randn(g, *shape, dtype=torch.float32):
    return torch.randn(*shape, generator=g, device="cuda").to(dtype)


def close(got, want, scale=None):
    got, want = got.float(), want.float()
    bound = ULP * (want.abs() if scale is None else scale.float()) + 1e-30
    assert torch.equal(got.isnan(), want.isnan())
    ok = ((got - want).abs() <= bound) | got.isnan() | (got == want)
    assert bool(ok.all()), float(((got - want).abs() / bound).nan_to_num().max())


# one thread's row, a ragged vector tail, no vectors, the last row kept in
# registers, the first that is not, one more than that
@pytest.mark.parametrize("rows,D", [(1, 4), (3, 36), (2, 37), (5, 1000), (7, 4096), (2, 4100), (2, 8209)])
def test_norms_and_additions(rows, D):
    g = gen(D)
    h, o, w = randn(g, rows, D), randn(g, rows, D, dtype=torch.bfloat16), randn(g, D, dtype=torch.bfloat16)
    close(K.rms_norm(h, w, 1e-6), _rms_norm(h, w, 1e-6).to(torch.bfloat16))
    h2, x = K.add_rms_norm(h, o, w, 1e-6)
    assert torch.equal(h2, h + o.float())
    close(x, _rms_norm(h2, w, 1e-6).to(torch.bfloat16))
    assert torch.equal(K.add_(h.clone(), o), h + o.float())
    assert torch.equal(K.to_bf16(h), h.to(torch.bfloat16))
    # rows that hold an infinity, a NaN, only zeros
    h[0, 0] = float("inf")
    h[-1, -1] = float("nan")
    close(K.rms_norm(h, w, 1e-6), _rms_norm(h, w, 1e-6).to(torch.bfloat16))
    assert not K.rms_norm(torch.zeros_like(h), w, 1e-6).any()


@pytest.mark.parametrize("rows,F", [(1, 4), (3, 260), (2, 1023), (2, 1028), (70000, 8)])
def test_silu_product(rows, F):
    y = randn(gen(F), rows, 2 * F, dtype=torch.bfloat16) * 8
    y[0, 0], y[-1, 1] = float("-inf"), -200.0
    gate, up = y[:, :F].contiguous(), y[:, F:].contiguous()
    want = (torch.nn.functional.silu(gate.float()) * up.float()).to(torch.bfloat16)
    close(K.silu_mul_joined(y), want)
    close(K.silu_mul(gate, up), want)


def both(model, h, pos):
    """qkv through the kernels and through torch (which a gradient asks for)."""
    assert model._kernels(0, h, pos)
    ours = model.qkv(0, h, pos)
    hg = h.clone().requires_grad_()
    assert not model._kernels(0, hg, pos)
    return ours, [t.detach() for t in model.qkv(0, hg, pos)]


@pytest.mark.parametrize("hq,hkv,d,D,F,rows", [(1, 1, 64, 64, 100, 1), (7, 1, 128, 260, 96, 5), (8, 2, 64, 256, 512, 33),
                                               (12, 4, 256, 520, 36, 9), (32, 8, 128, 4096, 384, 40)])
def test_layer_pieces(hq, hkv, d, D, F, rows):
    model = RandomDecoder(DecoderDims(1, hq, hkv, d, D, F, 77), seed=1)
    g = gen(d)
    w = model.layers[0]
    for n in ("in_norm", "q_norm", "k_norm", "post_norm"):
        w[n].copy_(1 + 0.1 * randn(g, w[n].numel()))
    h = randn(g, rows, D)
    pos = torch.randint(0, 100000, (rows,), generator=g, device="cuda")
    assert K.joined(w["wq"], w["wk"], w["wv"]) is not None and K.joined(w["w_gate"], w["w_up"]) is not None

    def check():
        (q, k, v), (qt, kt, vt) = both(model, h, pos)
        # the projections' own sums may round to the next bf16, which the
        # head's norm then scales: a few units of the head's largest values
        for a, b in ((q, qt), (k, kt), (v, vt)):
            assert a.is_contiguous() and a.shape == b.shape and a.dtype is b.dtype
            close(a, b, scale=2 * b.abs().amax(-1, keepdim=True).expand_as(b))
        attn = randn(g, rows, hq, d)
        want = model.block_out(0, h.clone().requires_grad_(), attn).detach()
        for a in (attn, attn.to(torch.bfloat16)):
            got = model.block_out(0, h, a)
            assert (got - want).abs().max() <= 4 * ULP * (want - h).abs().max()
        lt = model.logits(h.clone().requires_grad_()).detach()
        close(model.logits(h), lt, scale=lt.abs().amax(-1, keepdim=True).expand_as(lt))
        close(model.logits(h[0]), lt[0], scale=lt[0].abs().amax().expand_as(lt[0]))

    check()
    # weights of one's own: the matrices are no longer one
    w["wk"], w["w_up"] = w["wk"] * 2, w["w_up"].clone()
    assert K.joined(w["wq"], w["wk"], w["wv"]) is None and K.joined(w["w_gate"], w["w_up"]) is None
    check()
    # further leading dimensions, other position types
    q1, k1, v1 = model.qkv(0, h[None].expand(2, rows, D).contiguous(), pos.int()[None].expand(2, rows).contiguous())
    q0, k0, v0 = model.qkv(0, h, pos.float())
    for a, b in ((q1, q0), (k1, k0), (v1, v0)):
        close(a[1], b, scale=2 * b.abs().amax(-1, keepdim=True).expand_as(b))


def test_rope_angles_match_torch_bit_for_bit():
    """With unit rows (rms 1 exactly) only the rotation is left, whose
    operations and order are torch's."""
    model = RandomDecoder(DecoderDims(1, 1, 1, 128, 128, 8, 8), seed=0)
    w = model.layers[0]
    eye = torch.eye(128, device="cuda", dtype=torch.bfloat16)
    for n in ("wq", "wk", "wv"):
        w[n].copy_(eye)
    h = torch.ones(300, 128, device="cuda") * (torch.arange(128, device="cuda") % 2 * 2 - 1)
    pos = torch.arange(300, device="cuda") * 337
    (q, k, v), (qt, kt, vt) = both(model, h, pos)
    assert torch.equal(v, vt)
    assert (q != qt).float().mean() < 1e-3 and (k != kt).float().mean() < 1e-3
    close(q, qt, scale=torch.ones_like(qt))


def test_transforms_modes_and_other_types_take_the_torch_path():
    model = RandomDecoder(DecoderDims(1, 4, 2, 64, 128, 64, 50), seed=0)
    h, pos = randn(gen(), 6, 128), torch.arange(6, device="cuda")
    want = model.qkv(0, h, pos)[0]
    assert not model._kernels(0, h.double(), pos) and not model._kernels(0, h[:0], pos[:0])
    assert not model._kernels(0, h, pos[:1]) and not model._kernels(0, h.t().contiguous().t(), pos)
    with torch.autocast("cuda", dtype=torch.float16):
        assert not model._kernels(0, h, pos)
    per_row = torch.func.vmap(lambda r, p: model.qkv(0, r[None], p[None])[0][0])(h, pos)
    close(per_row, want, scale=2 * want.abs().amax(-1, keepdim=True).expand_as(want))
    _, tangent = torch.func.jvp(lambda x: model.logits(x), (h,), (h,))
    assert tangent.abs().max() > 0


def test_compilers_and_tracers_see_the_torch_expressions():
    """A whole graph without a break, a trace and a proxy's graph, each of
    which runs other inputs as the torch expressions do (bit for bit)."""
    from torch.fx.experimental.proxy_tensor import make_fx
    model = RandomDecoder(DecoderDims(1, 4, 2, 64, 128, 64, 50), seed=0)
    h, other, attn, pos = randn(gen(), 6, 128), randn(gen(1), 6, 128), randn(gen(2), 6, 4, 64), torch.arange(6, device="cuda")
    pieces = (lambda x: model.qkv(0, x, pos)[0], lambda x: model.block_out(0, x, attn), lambda x: model.logits(x))
    k, v = (torch.zeros(1, 2, 6, 64, device="cuda", dtype=torch.bfloat16) for _ in range(2))
    for f in pieces:
        want = f(other.clone().requires_grad_()).detach()
        with torch.no_grad():
            torch._dynamo.reset()
            for g in (torch.compile(f, backend="eager", fullgraph=True), torch.jit.trace(f, (h,), check_trace=False),
                      make_fx(f)(h)):
                assert torch.equal(g(other), want)
    torch._dynamo.reset()
    assert model.prefill(pos, k, v).isfinite().all()


def test_tensors_whose_values_are_not_at_their_address_take_the_torch_path():
    model = RandomDecoder(DecoderDims(1, 4, 2, 64, 128, 64, 50), seed=0)
    h, pos = randn(gen(), 6, 128), torch.arange(6, device="cuda")
    negated, nothing = torch._neg_view(h), torch._efficientzerotensor((6, 128), device="cuda")
    for x in (negated, nothing):
        assert not model._kernels(0, x, pos) and not model._kernels(0, x) and not K.plain((x,), ())
    for got, want in zip(model.qkv(0, negated, pos), model.qkv(0, -h, pos)):
        close(got, want, scale=2 * want.abs().amax(-1, keepdim=True).expand_as(want))
    weight = torch._neg_view(model.layers[0]["wo"])
    assert not K.plain((h,), (weight,))


def test_an_mlp_of_no_width():
    """The torch expressions add nothing for it; a kernel has nothing to launch."""
    model = RandomDecoder(DecoderDims(1, 2, 1, 64, 128, 0, 50), seed=0)
    h, attn = randn(gen(), 6, 128), randn(gen(1), 6, 2, 64)
    want = model.block_out(0, h.clone().requires_grad_(), attn).detach()
    close(model.block_out(0, h, attn), want, scale=want.abs().amax().expand_as(want))


@pytest.mark.parametrize("hq,hkv,d,T", [(1, 1, 64, 1), (6, 2, 128, 77), (4, 4, 256, 130)])
def test_prefill_into_stores_and_into_copies(hq, hkv, d, T):
    """Straight into contiguous bf16 stores, and through copies into others."""
    model = RandomDecoder(DecoderDims(2, hq, hkv, d, 192, 320, 60), seed=2)
    tokens = torch.randint(0, 60, (T,), generator=gen(T), device="cuda")
    k, v = (torch.zeros(2, hkv, T, d, device="cuda", dtype=torch.bfloat16) for _ in range(2))
    kf, vf = (torch.zeros(2, hkv, T, d, device="cuda") for _ in range(2))
    want = model.prefill(tokens, kf, vf)
    got = model.prefill(tokens, k, v)
    assert torch.equal(k.float(), kf) and torch.equal(v.float(), vf) and torch.equal(got, want)


def test_prefill_gives_a_block_out_of_ones_own_fp32():
    dims, kinds = DecoderDims(2, 4, 2, 64, 128, 64, 50), []

    class Own(RandomDecoder):
        def block_out(self, l, h, attn):
            kinds.append(attn.dtype)
            return super().block_out(l, h, attn)

    tokens = torch.arange(9, device="cuda")
    stores = [torch.zeros(2, 2, 9, 64, device="cuda", dtype=torch.bfloat16) for _ in range(2)]
    assert torch.equal(Own(dims).prefill(tokens, *stores), RandomDecoder(dims).prefill(tokens, *stores))
    assert kinds == [torch.float32] * 2


def test_prefill_writes_its_stores_as_torch_does():
    """A graph that saved a store sees that it was written since; a store of
    inference mode is refused outside it."""
    model = RandomDecoder(DecoderDims(1, 2, 1, 64, 128, 64, 50), seed=0)
    tokens = torch.arange(9, device="cuda")
    k, v = (torch.zeros(1, 1, 9, 64, device="cuda", dtype=torch.bfloat16) for _ in range(2))
    for store in (k, v):
        x = torch.ones(64, device="cuda", dtype=torch.bfloat16, requires_grad=True)
        y = (x * store).sum()
        model.prefill(tokens, k, v)
        with pytest.raises(RuntimeError, match="modified by an inplace operation"):
            y.backward()
    with torch.inference_mode():
        ki, vi = torch.zeros_like(k), torch.zeros_like(v)
        model.prefill(tokens, ki, vi)
        assert torch.equal(ki, k) and torch.equal(vi, v)
    for stores in ((ki, v), (k, vi)):
        with pytest.raises(RuntimeError, match="inference tensor"):
            model.prefill(tokens, *stores)


def gemm(mode, x, w0, w1=None, h=None):
    M, k, N = x.shape[0], x.shape[1], w0.shape[0]
    y = torch.full((M + 1, N), float("nan"), dtype=torch.float32 if mode == 1 else torch.bfloat16, device="cuda")
    p = [t.data_ptr() if t is not None else None for t in (x, w0, w1, h, y)]
    assert K.lib().decoder_gemm(mode, *p, M, N, k, torch.cuda.current_stream().cuda_stream) == 0
    K.check_device_error()
    assert bool(y[M].isnan().all())             # nothing past the last row
    return y[:M].double()


# a pair of CTAs per tile and clusters of up to three; ragged rows, features and
# K; gate and up of one matrix or of two
@pytest.mark.parametrize("M", [1, 15, 16, 17, 64, 100, 128, 129, 256, 257, 400])
@pytest.mark.parametrize("N,k", [(1, 8), (130, 72), (640, 1000), (4096, 512), (2000, 4096), (20000, 136), (256, 12288)])
def test_fused_projections(M, N, k):
    """fp32 sums of K exact products, each addition of 16 of them truncated at
    2^-23 of the largest partial sum at most; then the output's own rounding."""
    g = gen(M + N + k)
    x, wa, wb = (randn(g, n, k, dtype=torch.bfloat16) for n in (M, N, N))
    wa, wb = ((w.float() * k ** -0.5).bfloat16() for w in (wa, wb))
    h = randn(g, M, N)
    a, b = (x.double() @ w.double().t() for w in (wa, wb))
    ma, mb = (x.double().abs() @ w.double().abs().t() for w in (wa, wb))
    e = (k / 16 + 12) * 2.0 ** -23
    assert bool(((gemm(0, x, wa) - a).abs() <= e * ma + 2.0 ** -8 * a.abs() + 1e-30).all())
    assert bool(((gemm(1, x, wa, h=h) - (h.double() + a)).abs() <= e * ma + 2.0 ** -23 * (h.double() + a).abs()).all())
    assert bool(((gemm(1, x, wa) - a).abs() <= e * ma + 2.0 ** -23 * a.abs()).all())
    s = torch.nn.functional.silu(a) * b
    # (|silu'| <= 1.1)
    bound = 1.1 * e * ma * (b.abs() + e * mb) + e * mb * a.abs() + (2.0 ** -8 + 2.0 ** -20) * s.abs() + 1e-30
    gate_up, up_gate = torch.cat([wa, wb]), torch.cat([wb, wa])
    for gate, up in ((gate_up[:N], gate_up[N:]), (up_gate[N:], up_gate[:N])):
        assert bool(((gemm(2, x, gate, up) - s).abs() <= bound).all())


def test_fused_silu_over_its_range():
    """Gates far below zero too, where e^-g nears and passes fp32's largest value
    (silu is 0 from there on, as torch's of fp32 is): the output's rounding to
    bf16, whose eight significant bits put it within 2^-8, and no more.  Gates of bf16 by weights of one and ups of one are exact."""
    g = torch.linspace(-95, 95, 64 * 64, device="cuda").bfloat16().view(64, 64)
    g[0, :12] = torch.tensor([-20, -80, -86.5, -87, -87.5, -88, -88.5, -89, -90, -200, -1e30, 1e30])
    x = torch.cat([g, torch.ones_like(g)], 1)
    eye, no = torch.eye(64, device="cuda", dtype=torch.bfloat16), torch.zeros(64, 64, device="cuda", dtype=torch.bfloat16)
    up = no.clone()
    up[:, 0] = 1
    got = gemm(2, x, torch.cat([eye, no], 1), torch.cat([no, up], 1))
    want = g.double() / (1 + torch.exp(-g.double()))
    want = torch.where(g < -88.7, 0.0, want)
    assert bool(((got - want).abs() <= (2.0 ** -8 + 2.0 ** -20) * want.abs()).all())


def test_fused_projection_rows_are_independent():
    """An infinity or NaN in a row of x stays in that row, the same bits with
    or without it; the same call twice gives the same bits."""
    g = gen(3)
    x, w = randn(g, 20, 1024, dtype=torch.bfloat16), randn(g, 300, 1024, dtype=torch.bfloat16)
    want = gemm(0, x, w)
    assert torch.equal(gemm(0, x, w), want)
    x[7, 100], x[12, 0] = float("inf"), float("nan")
    got = gemm(0, x, w)
    rest = [r for r in range(20) if r not in (7, 12)]
    assert torch.equal(got[rest], want[rest])
    assert not bool(got[7].isfinite().any()) and bool(got[12].isnan().all())


def test_fused_projections_behind_one_another():
    """Launches of every kind of shape in a row, so that one's CTAs come to SMs
    that another's have just left: each gives the bits it gives alone."""
    g = gen(9)
    cases = []
    for M, N, k in ((1, 4096, 4096), (16, 640, 1000), (64, 6144, 512), (257, 4096, 512), (400, 20000, 136), (3, 130, 72)):
        x, w = randn(g, M, k, dtype=torch.bfloat16), randn(g, N, k, dtype=torch.bfloat16)
        cases.append((x, w, gemm(1, x, w).float()))
    outs = []
    for i in range(60):
        x, w, want = cases[i * 5 % len(cases)]
        y = torch.empty_like(want)
        assert K.lib().decoder_gemm(1, x.data_ptr(), w.data_ptr(), None, None, y.data_ptr(), *want.shape, x.shape[1],
                                    torch.cuda.current_stream().cuda_stream) == 0
        outs.append((y, want))
    K.check_device_error()
    for y, want in outs:
        assert torch.equal(y, want)


# one row; a tile of rows, two; shares of K; more tiles than pairs of CTAs;
# many rows; rows of the MLP that TMA does not take
@pytest.mark.parametrize("rows,ffn", [(1, 1544), (128, 1544), (257, 1544), (300, 12288), (1030, 1544), (9000, 12288),
                                      (40, 1541)])
def test_layer_on_fused_projections_and_on_the_librarys(rows, ffn):
    """A half of the layer is one call on the fused projections or the
    library's GEMMs with kernels between; both meet the torch expressions."""
    model = RandomDecoder(DecoderDims(1, 6, 2, 128, 1024, ffn, 40), seed=4)
    g = gen(rows)
    assert K.lib().decoder_scratch_bytes(0, rows, 1024, 768, 1280, 0) > 0
    assert (K.lib().decoder_scratch_bytes(1, rows, 1024, 768, 0, ffn) > 0) == (ffn % 8 == 0)
    h, pos, attn = randn(g, rows, 1024), torch.arange(rows, device="cuda"), randn(g, rows, 6, 128)
    (q, k, v), (qt, kt, vt) = both(model, h, pos)
    for a, b in ((q, qt), (k, kt), (v, vt)):
        close(a, b, scale=2 * b.abs().amax(-1, keepdim=True).expand_as(b))
    want = model.block_out(0, h.clone().requires_grad_(), attn).detach()
    kept = h.clone()
    got = model.block_out(0, h, attn)
    assert torch.equal(h, kept) and got.data_ptr() != h.data_ptr()
    assert (got - want).abs().max() <= 4 * ULP * (want - h).abs().max()
    K.check_device_error()


def assert_causal(got, q, k, v, scale):
    """Probabilities and outputs are rounded to bf16, whose eight significant
    bits put a rounded value within 2^-8 of it each time; a score of d
    exact products is off by at most 2^-21 of the sum of their magnitudes, and
    its probability by as much again."""
    G, T = q.shape[1] // k.shape[0], q.shape[0]
    kd, vd = (x.double().repeat_interleave(G, 0) for x in (k, v))
    qd = q.double().transpose(0, 1)
    z = (qd @ kd.transpose(1, 2) * scale).masked_fill(torch.ones(T, T, device="cuda").triu(1).bool(), float("-inf"))
    w = torch.softmax(z, -1)
    want, size = (w @ vd).transpose(0, 1), (w @ vd.abs()).transpose(0, 1)
    mag = (qd.abs() @ kd.abs().transpose(1, 2) * abs(scale)).amax(-1).t()[..., None]
    bound = (2.0 ** -8 + 2 * 2.0 ** -21 * mag + 2.0 ** -19) * size
    bound = bound + 2.0 ** -8 * (want.abs() + bound) + 1e-30
    assert bool(((got.double() - want).abs() <= bound).all())


# one row; edges of a key block and of a tile of rows; many tiles; every head
# dim, with one and more query heads to a kv head
@pytest.mark.parametrize("T", [1, 63, 64, 65, 127, 128, 129, 200, 1000])
@pytest.mark.parametrize("hq,hkv,d", [(3, 3, 64), (8, 2, 128), (7, 1, 256)])
def test_causal_attention(T, hq, hkv, d):
    g = gen(T + d)
    q, k, v = randn(g, T, hq, d), randn(g, hkv, T, d), randn(g, hkv, T, d)
    k[:, -1] *= 6                     # a later maximum far above the earlier ones
    q, k, v = q.bfloat16(), k.bfloat16(), v.bfloat16()
    got = K.causal(q, k, v, d ** -0.5)
    K.check_device_error()
    assert_causal(got, q, k, v, d ** -0.5)


# scales that the model's caller may set, two that fp32 holds as zero or denormal
@pytest.mark.parametrize("scale", [0.0, -0.0, 1e-50, 1e-40, -1e-3, -0.125, -1.0])
@pytest.mark.parametrize("hq,hkv,d", [(2, 1, 64), (4, 2, 128), (2, 2, 256)])
def test_causal_attention_at_any_scale(hq, hkv, d, scale):
    """As with a positive scale (the bound is test_causal_attention's)."""
    T, g = 200, gen(d)
    q, k, v = (randn(g, *s, dtype=torch.bfloat16) for s in ((T, hq, d), (hkv, T, d), (hkv, T, d)))
    got = K.causal(q, k, v, scale)
    K.check_device_error()
    assert_causal(got, q, k, v, scale)


def test_causal_attention_rows_do_not_see_later_ones():
    g = gen(5)
    q, k, v = (randn(g, *s, dtype=torch.bfloat16) for s in ((300, 4, 128), (2, 300, 128), (2, 300, 128)))
    want = K.causal(q, k, v, 0.1)
    k[:, 256:], v[:, 256:] = float("inf"), float("nan")
    assert torch.equal(K.causal(q, k, v, 0.1)[:256], want[:256])


# some keys of the first block, all of it, more, and more than a tile of rows
@pytest.mark.parametrize("ruled_out", [10, 64, 70, 200])
@pytest.mark.parametrize("d", [64, 128, 256])
def test_causal_attention_over_keys_that_are_ruled_out(ruled_out, d):
    """A key whose score is -inf weighs nothing, also where a row has met no
    other yet; a row that meets no other at all gives zeros."""
    g = gen(d)
    q, k, v = (randn(g, *s, dtype=torch.bfloat16) for s in ((260, 2, d), (1, 260, d), (1, 260, d)))
    q[:, :, 0] = 1
    k[:, :ruled_out, 0] = float("-inf")
    got = K.causal(q, k, v, d ** -0.5)
    K.check_device_error()
    assert not bool(got[:ruled_out].any())
    assert_causal(got[ruled_out:], q[ruled_out:], k[:, ruled_out:], v[:, ruled_out:], d ** -0.5)


@pytest.mark.parametrize("hq,hkv,d", [(32, 8, 64), (32, 8, 128), (16, 2, 256)])
def test_causal_attention_is_the_same_every_time(hq, hkv, d):
    """Every SM full, its CTAs at every distance from one another."""
    g = gen(d)
    q, k, v = (randn(g, *s, dtype=torch.bfloat16) for s in ((1500, hq, d), (hkv, 1500, d), (hkv, 1500, d)))
    want = K.causal(q, k, v, d ** -0.5)
    for _ in range(20):
        assert torch.equal(K.causal(q, k, v, d ** -0.5), want)
    K.check_device_error()


# one tile per pair of CTAs and shares of K; tiles by waves, with a tail; the
# library's head (more than 256 rows)
@pytest.mark.parametrize("rows", [9, 300])
def test_a_captured_graph_of_the_pieces(rows):
    """Replayed on other inputs in the same buffers: the eager calls' bits."""
    model = RandomDecoder(DecoderDims(1, 6, 2, 128, 1024, 9000, 500), seed=4)
    g = gen(rows)
    h, attn, pos = randn(g, rows, 1024), randn(g, rows, 6, 128), torch.arange(rows, device="cuda")
    tokens = torch.randint(0, 500, (rows,), generator=g, device="cuda")
    k, v = (torch.zeros(1, 2, rows, 128, device="cuda", dtype=torch.bfloat16) for _ in range(2))

    def pieces():
        return (*model.qkv(0, h, pos), model.block_out(0, h, attn), model.logits(h), model.prefill(tokens, k, v), k, v)

    with torch.no_grad():
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            pieces()
        torch.cuda.current_stream().wait_stream(side)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            out = pieces()
        for _ in range(3):
            for x, new in ((h, randn(g, rows, 1024)), (attn, randn(g, rows, 6, 128)), (pos, pos + 77),
                           (tokens, tokens.flip(0).clone())):
                x.copy_(new)
            want = [t.clone() for t in pieces()]
            for t in out:
                t.fill_(float("nan"))
            graph.replay()
            assert all(torch.equal(a, b) for a, b in zip(out, want))
    K.check_device_error()


def test_two_streams_at_once():
    """Layers on two streams, each in its own order, with the scratch and the
    outputs of many calls in flight: the bits of each alone."""
    models = [RandomDecoder(DecoderDims(1, 8, 2, 128, 2048, 5000, 700), seed=i) for i in range(2)]
    g = gen(6)
    work = [[(randn(g, n, 2048), randn(g, n, 8, 128), torch.arange(n, device="cuda")) for n in rows]
            for rows in ((1, 40, 300, 700), (513, 7, 130, 256))]

    def pieces(m, h, attn, pos):
        q, k, v = m.qkv(0, h, pos)
        return (q, k, v, m.block_out(0, h, attn), m.logits(h),
                K.causal(q, k.transpose(0, 1).contiguous(), v.transpose(0, 1).contiguous(), 0.1))

    want = [[pieces(m, *w) for w in ws] for m, ws in zip(models, work)]
    streams = [torch.cuda.Stream() for _ in range(2)]
    torch.cuda.synchronize()
    got = []
    for i in range(40):
        for m, ws, wants, stream in zip(models, work, want, streams):
            with torch.cuda.stream(stream):
                got.append((pieces(m, *ws[i % 4]), wants[i % 4]))
    K.check_device_error()
    for a, b in got:
        assert all(torch.equal(x, y) for x, y in zip(a, b))


@pytest.mark.skipif(torch.cuda.device_count() < 2, reason="one device")
def test_a_second_device():
    """Both devices of a process, one after the other."""
    outs = []
    for dev in range(2):
        with torch.cuda.device(dev):
            model = RandomDecoder(DecoderDims(1, 4, 2, 128, 256, 512, 60), device=f"cuda:{dev}")
            k, v = (torch.zeros(1, 2, 70, 128, device="cuda", dtype=torch.bfloat16) for _ in range(2))
            outs.append(model.prefill(torch.arange(70, device="cuda") % 60, k, v).cpu())
            K.check_device_error()
    assert torch.equal(*outs)


def test_the_error_check_waits_for_every_stream():
    """Launches on a side stream, whose streams torch makes non-blocking, may
    still set the word."""
    K.check_device_error()
    side, done = torch.cuda.Stream(), torch.cuda.Event()
    with torch.cuda.stream(side):
        torch.cuda._sleep(200_000_000)          # some 0.1 s
        done.record()
    assert not done.query()
    K.check_device_error()
    assert done.query()
