"""Launch shapes of the decoder's fused projections (host arithmetic): what a
CTA puts where stays inside what the launch gives it."""
import ctypes

import pytest

from paper_2605_30574_gb300 import build as B
from paper_2605_30574_gb300 import decoder as K


@pytest.fixture(scope="module")
def lib():
    B.build()
    return K.lib()


def test_every_launch_fits(lib):
    out = (ctypes.c_long * 15)()
    for mode in (0, 1, 2):
        for room in ((76, 36, 23, 15), (74, 36, 22, 14), (10, 4, 0, 0), (1, 0, 0, 0)):
            resident = (ctypes.c_int * 4)(*room)
            for M in [*range(1, 130), *range(130, 514, 17), 255, 256, 257, 512, 513, 1024, 4000, 65536]:
                for N in (1, 8, 127, 128, 129, 640, 2000, 4096, 6144, 12288, 40000, 151936):
                    for k in (8, 64, 72, 504, 512, 1000, 1024, 4096, 12288, 20000):
                        assert lib.decoder_gemm_plan(mode, M, N, k, resident, out) == 0
                        mp, kblocks, split, tiles, tiles_m, clusters, stages, stage, cols, bufs, traded, smem, tail, tail_mp, tail_m = out
                        feat = 128 if mode == 2 else 256
                        assert mp % 32 == 0 and 32 <= mp <= 256 and tiles_m * mp >= M > (tiles_m - 1) * mp
                        assert tiles * feat >= N > (tiles - 1) * feat and kblocks * 64 >= k > (kblocks - 1) * 64
                        # every pair has K blocks; shares of K are of one tile, all of them resident
                        assert 1 <= split <= 4 and kblocks >= split and 1 <= clusters <= max(room[split - 1], 1)
                        assert clusters == tiles * tiles_m if split > 1 else clusters <= tiles * tiles_m
                        # an accumulator to spare where a pair has a second tile
                        assert cols <= 512 and cols & (cols - 1) == 0 and mp * bufs <= cols
                        assert bufs == (2 if tiles * tiles_m > clusters else 1)
                        # the tail: smaller tiles, of all rows, that fill one wave at the most
                        assert 0 <= tail <= tiles and tail_mp % 32 == 0 and 32 <= tail_mp <= mp
                        if tail < tiles:
                            waves = tiles * tiles_m // clusters
                            assert split == 1 and tail_m * tail_mp >= M > (tail_m - 1) * tail_mp and bufs == 2
                            assert waves * clusters < tail * tiles_m + (tiles - tail) * tail_m <= (waves + 1) * clusters
                        # a stage holds W's and half of x's block; the ring the sums that the pairs trade
                        assert stage == 16384 + mp * 64 and stage % 1024 == 0 and stages >= 2
                        chunks = mp // 16
                        last = ((split - 1) * -(-chunks // split) + (chunks - 1) // split + 1) * 8192
                        assert traded >= (last if split > 1 else 0) and traded <= stages * stage
                        # a warp's chunks of a share, two warps to them, are four at the most
                        assert split == 1 or -(-(-(-chunks // split)) // 2) <= 4
                        # one CTA to an SM (and its TMEM)
                        assert smem == stages * stage + 1024 <= 226 * 1024 and 2 * (smem + 1024) > 228 * 1024
    room = (ctypes.c_int * 4)(76, 36, 23, 15)
    for bad in ((0, 0, 8, 8), (0, 65537, 8, 8), (0, 1, 0, 8), (0, 1, 8, 12), (3, 1, 8, 8), (-1, 1, 8, 8)):
        assert lib.decoder_gemm_plan(*bad, room, out) != 0


def test_misaligned_words_are_refused_before_any_launch(lib):
    """Every pointer and stride that is read or written in words of d / 64
    elements, one at a time off by an element."""
    for d in (128, 256):
        ok = [1 << 20] * 6                       # (never read: each call is refused)
        norms = [1 << 20] * 2

        def post(ptrs, strides, norms):
            return lib.decoder_qkv_post(*ptrs, (ctypes.c_long * 9)(*strides), *norms, 1 << 20, 1 << 20, 0, 1, 1, 1, d, 1e-6, 0)

        def off(values, i, by):
            return [v + by * (j == i) for j, v in enumerate(values)]

        for i in range(6):
            assert post(off(ok, i, 2), [d] * 9, norms) == 1
        for i in range(9):
            assert post(ok, off([d] * 9, i, 1), norms) == 1
        for i in range(2):
            assert post(ok, [d] * 9, off(norms, i, 2)) == 1
            one = off(norms, i, 2)
            assert lib.decoder_qkv(1 << 20, 1 << 20, 1 << 20, 1 << 20, *ok[:3], (ctypes.c_long * 6)(*[d] * 6), *one,
                                   1 << 20, 1 << 20, 0, 1, 64, 1, 1, d, 1e-6, 0) == 1
    assert lib.decoder_qkv_post(*[1 << 20] * 6, (ctypes.c_long * 9)(*[96] * 9), *[1 << 20] * 4, 0, 1, 1, 1, 96, 1e-6, 0) == 1
