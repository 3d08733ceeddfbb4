"""The generated-span pass by itself -- ZERO donors everywhere, so a row's
prompt span is the closed form -- at every group size and head dim, at the
edges of its 16-key blocks and key splits, against fp64.

Bound: the pass computes in fp32.  A logit of d exact products summed in fp32
is off by at most 2^-22 of the sum of their magnitudes (a chain of two
products of the tensor core and seven additions at the most, each within
2^-24 to 2^-23); a probability by that times ln 2 in log2 units, and by 2^-21
for exp2; the weighted sum of n values in chains of at most n / 16 + 4
additions by (n / 16 + 4) 2^-24 of the largest value."""
import pytest
import torch

from paper_2605_30574_gb300 import build as B
from paper_2605_30574_gb300 import splice as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    B.build()


class Span:
    def __init__(self, G, d, t, cells, hkv=2, T=None, seed=0):
        g = torch.Generator(device="cuda")
        g.manual_seed(seed)
        r = lambda *s: torch.randn(*s, generator=g, device="cuda").bfloat16()  # noqa: E731
        self.G, self.d, self.t, self.n, self.hkv, T = G, d, t, cells, hkv, T or t
        self.ks, self.vs, self.q = r(cells, 2, hkv, T, d), r(cells, 2, hkv, T, d), r(cells, hkv * G, d)
        self.q = (self.q.float() * d ** -0.5).bfloat16()
        self.kn, self.vn, self.kc = r(cells, hkv, d), r(cells, hkv, d), r(1, 2, hkv, 3, d)
        shape = dict(num_layers=2, num_q_heads=hkv * G, num_kv_heads=hkv, head_dim=d, sliding_window=0,
                     global_every=0, sm_scale=1.0)
        self.desc = S.splice_desc_create(shape, 1, 3, (S.DONOR_ZERO,), [(0, 0, 0, 0)] * cells, T)
        self.ws = torch.empty(S.splice_workspace_bytes(self.desc), dtype=torch.uint8, device="cuda")
        self.out = torch.full((cells, hkv * G, d), float("nan"), device="cuda")

    def step(self):
        S.spliced_decode_step(self.desc, 1, self.t, self.q, self.kn, self.vn, self.kc, self.kc, None, None, self.ks,
                              self.vs, self.out, self.ws)
        S.splice_check_device_error(self.desc)
        return self.out

    def exact(self):
        """(output, bound) with the step's own entry in place."""
        K, V = self.ks[:, 1, :, :self.t].double(), self.vs[:, 1, :, :self.t].double()
        K[:, :, -1], V[:, :, -1] = self.kn.double(), self.vn.double()
        x = self.q.double().unflatten(1, (self.hkv, self.G))
        z = torch.einsum("bhgd,bhnd->bhgn", x, K)
        z = torch.cat([z.new_zeros(*z.shape[:-1], 3), z], -1)                  # the ZERO span's three keys
        out = torch.einsum("bhgn,bhnd->bhgd", torch.softmax(z, -1)[..., 3:], V)
        mag = torch.einsum("bhgd,bhnd->bhgn", x.abs(), K.abs()).amax(-1, keepdim=True)
        rel = 2 * 2.0 ** -22 * mag + 2.0 ** -20 + (self.t / 16 + 4) * 2.0 ** -24
        bound = rel * V.abs().amax((-2, -1), keepdim=True)
        return out.flatten(1, 2), bound.expand_as(out).flatten(1, 2)


@pytest.mark.parametrize("d", [64, 128, 256])
@pytest.mark.parametrize("G", [1, 2, 3, 4, 5, 7, 8, 9, 12, 16])
def test_every_group_size(G, d):
    # one entry; a block short of one, whole, and one over; several splits,
    # the last ragged; more items than warps
    for t, cells in ((1, 3), (15, 2), (16, 2), (17, 2), (64, 1), (209, 3), (530, 2), (33, 700), (5, 1000)):
        s = Span(G, d, t, cells, seed=t)
        want, bound = s.exact()
        err = (s.step().double() - want).abs()
        assert bool((err <= bound).all()), (G, d, t, float((err / bound).max()))
        assert torch.equal(s.ks[:, 1, :, t - 1], s.kn) and torch.equal(s.vs[:, 1, :, t - 1], s.vn)


@pytest.mark.parametrize("G,d", [(1, 128), (2, 256), (4, 64), (5, 128), (8, 256), (16, 128)])
def test_infinities_and_nans(G, d):
    """An infinite value makes only its own dimension infinite, a NaN only its
    own NaN, in the store and in the step's own entry; an infinite key weighs
    nothing in the rows it is negative for (the rows it is positive for have
    no softmax, and are not looked at)."""
    t = 70
    s = Span(G, d, t, 6, seed=5)
    s.q = (s.q.float() * 0.1).bfloat16()
    clean, bound = s.exact()
    inf, nan = float("inf"), float("nan")
    s.vs[0, 1, :, 20, 3] = inf
    s.vs[1, 1, :, 33, d - 1] = nan
    s.vn[2, :, 7] = -inf
    s.vs[3, 1, :, 0, 5], s.vs[3, 1, :, 64, 5] = inf, -inf
    s.ks[4, 1, :, 11, 0] = inf
    out = s.step().double()
    close = (out - clean).abs() <= bound + 1e-6
    for cell, dim, what in ((0, 3, inf), (1, d - 1, nan), (2, 7, -inf), (3, 5, nan)):
        col = out[cell, :, dim]
        assert bool(col.isnan().all() if what != what else (col == what).all()), (cell, col)
        rest = torch.arange(d, device="cuda") != dim
        assert bool(close[cell][:, rest].all()), cell
    sign = s.q[4, :, 0]
    # the ruled-out key's weight is gone: compare without it
    K = torch.cat([s.ks[4, 1, :, :11], s.ks[4, 1, :, 12:t - 1], s.kn[4][:, None]], 1).double()
    V = torch.cat([s.vs[4, 1, :, :11], s.vs[4, 1, :, 12:t - 1], s.vn[4][:, None]], 1).double()
    z = torch.einsum("hgd,hnd->hgn", s.q[4].double().unflatten(0, (s.hkv, G)), K)
    z = torch.cat([z.new_zeros(*z.shape[:-1], 3), z], -1)
    want = torch.einsum("hgn,hnd->hgd", torch.softmax(z, -1)[..., 3:], V).flatten(0, 1)
    assert bool(((out[4] - want).abs() <= bound[4] + 1e-6)[sign < 0].all())
    assert bool(close[5].all())


def test_bf16_extremes():
    """Keys of the lowest bf16 value rule themselves out or in; large values
    stay finite."""
    s = Span(5, 128, 40, 2, seed=9)
    low = torch.finfo(torch.bfloat16).min
    s.q.zero_()
    s.q[:, :, 0] = 1.0
    s.ks[:, 1, :, 3] = 0
    s.ks[:, 1, :, 3, 0] = low
    s.vs[:, 1, :, 5] = 1e36
    want, _ = s.exact()
    out = s.step().double()
    assert bool(out.isfinite().all())
    assert bool(((out - want).abs() <= 1e-5 * want.abs().amax()).all())
