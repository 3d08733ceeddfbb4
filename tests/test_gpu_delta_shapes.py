"""The delta encoding at the edges of its rounds, clusters and rows: every
byte of the buffer's four parts against the definition in plain torch (bit
for bit: the encoding is a copy)."""
import pytest
import torch

from paper_2605_30574_gb300 import build as B
from paper_2605_30574_gb300 import splice as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    B.build()


def stores(P, Dst, N, H, Tp, d, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    bits = lambda *s: torch.randint(-2 ** 15, 2 ** 15, s, generator=g, device="cuda", dtype=torch.int16)  # noqa: E731
    kc, vc = bits(P, N, H, Tp, d), bits(P, N, H, Tp, d)
    kd, vd = (x[:, None].expand(P, Dst, N, H, Tp, d).clone() for x in (kc, vc))
    # per span: nothing, everything, or a share of the positions differs, by
    # one bit of one element of the K row, the V row or both
    share = torch.rand(P, Dst, N, H, 1, generator=g, device="cuda") * 1.6 - 0.3
    pick = torch.rand(P, Dst, N, H, Tp, generator=g, device="cuda") < share
    which = torch.randint(1, 4, pick.shape, generator=g, device="cuda")
    c = torch.randint(0, d, pick.shape, generator=g, device="cuda")
    one = torch.nn.functional.one_hot(c, d).to(torch.int16) << torch.randint(0, 15, (*pick.shape, 1), generator=g,
                                                                             device="cuda").to(torch.int16)
    kd ^= one * (pick & (which != 2))[..., None]
    vd ^= one * (pick & (which != 1))[..., None]
    return kc, vc, kd, vd, pick


def check(P, kinds, N, H, Tp, d, seed=0):
    Dst = sum(k != S.DONOR_ZERO for k in kinds)
    shape = dict(num_layers=N, num_q_heads=H, num_kv_heads=H, head_dim=d, sliding_window=0, global_every=0,
                 sm_scale=1.0)
    desc = S.splice_desc_create(shape, P, Tp, kinds, [(0, 0, 0, 0)], 2)
    kc, vc, kd, vd, pick = stores(P, Dst, N, H, Tp, d, seed)
    nbytes = S.splice_delta_bytes(desc)
    buf = torch.full((nbytes + 256,), 0xA5, dtype=torch.uint8, device="cuda")
    frac = S.splice_delta_build(desc, kc, vc, kd, vd, buf, delta_bytes=nbytes)
    torch.cuda.synchronize()
    al = lambda x: (x + 255) // 256 * 256  # noqa: E731
    spans, w32, rows = P * Dst * N * H, 4 * ((Tp + 127) // 128), P * Dst * N * H * Tp * d * 2
    count_off = al(spans * w32 * 4)
    k_off = al(count_off + spans * 4)
    v_off = al(k_off + rows)
    assert v_off + rows == nbytes and bool((buf[nbytes:] == 0xA5).all())
    flat = pick.view(spans, Tp)
    padded = torch.zeros(spans, w32 * 32, dtype=torch.int64, device="cuda")
    padded[:, :Tp] = flat
    words = (padded.view(spans, w32, 32) << torch.arange(32, device="cuda")).sum(-1)
    got = buf[:spans * w32 * 4].view(torch.int32).view(spans, w32).to(torch.int64) & 0xFFFFFFFF
    assert torch.equal(got, words)
    n = flat.sum(-1)
    assert torch.equal(buf[count_off:count_off + spans * 4].view(torch.int32).to(torch.int64), n)
    order = torch.argsort((~flat).to(torch.int8), dim=1, stable=True)           # encoded positions first, in order
    live = torch.arange(Tp, device="cuda")[None] < n[:, None]
    for off, src in ((k_off, kd), (v_off, vd)):
        want = torch.gather(src.view(spans, Tp, d), 1, order[..., None].expand(spans, Tp, d)) * live[..., None]
        assert torch.equal(buf[off:off + rows].view(torch.int16).view(spans, Tp, d), want.to(torch.int16))
    per = iter(pick.double().mean((0, 2, 3, 4)).tolist())
    for k, f in zip(kinds, frac):
        assert f == -1.0 if k == S.DONOR_ZERO else abs(f - next(per)) < 1e-6
    desc.close()


# a chunk is 128, 64 or 32 positions (d = 64, 128, 256), a round up to eight of them
@pytest.mark.parametrize("d", [64, 128, 256])
@pytest.mark.parametrize("Tp", [1, 3, 31, 33, 64, 127, 129, 257, 640, 1025, 2050])
def test_few_spans(d, Tp):
    check(1, (S.DONOR_BLANK, S.DONOR_ZERO, S.DONOR_SAME_ALGO), 2, 3, Tp, d, seed=Tp)


# 4096, 2400 and 960 spans: one, two and four CTAs per span on 152 SMs
@pytest.mark.parametrize("P,N,H", [(8, 16, 16), (5, 15, 16), (4, 8, 15)])
@pytest.mark.parametrize("d,Tp", [(64, 300), (128, 150), (256, 130)])
def test_many_spans(P, N, H, d, Tp):
    check(P, (S.DONOR_BLANK, S.DONOR_SAME_ALGO), N, H, Tp, d, seed=P)
