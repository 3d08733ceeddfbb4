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
    out = (ctypes.c_long * 10)()
    for mode in (0, 1, 2):
        parts = 2 if mode == 2 else 1
        for sms in (152, 148, 20, 1):
            for M in [*range(1, 130), *range(130, 514, 17), 255, 256, 257, 512, 513, 1024, 4000]:
                for N in (1, 8, 127, 128, 129, 640, 2000, 4096, 6144, 12288, 40000, 151936):
                    for k in (8, 64, 72, 504, 512, 1000, 1024, 4096, 12288, 20000):
                        takes = M <= 512 or -(-M // 256) * N * k * 2 <= 64 << 20
                        assert (lib.decoder_gemm_plan(mode, M, N, k, sms, out) == 0) == takes
                        if not takes:
                            continue
                        mp, kblocks, split, tiles, stages, stage, cols, traded, smem, tiles_m = out
                        assert mp % 16 == 0 and mp <= 256 and mp < M + 16 and (mp >= M if M <= 128 else mp > 64)
                        assert tiles_m * mp >= M > (tiles_m - 1) * mp
                        assert tiles * 128 >= N > (tiles - 1) * 128 and kblocks * 64 >= k > (kblocks - 1) * 64
                        per_sm = 2 if mp <= 128 else 1
                        assert 1 <= split <= 8 and (split == 1 or tiles * tiles_m * split <= per_sm * sms)
                        # every CTA of a cluster has K blocks, the accumulators columns
                        assert kblocks >= split and parts * mp <= cols and per_sm * cols <= 512 and cols & (cols - 1) == 0
                        # a stage holds W's and x's block; the ring the sums that the CTAs trade
                        assert stage >= parts * 16384 + mp * 128 and stage % 1024 == 0 and stages >= 2
                        chunks = mp // 16
                        last = ((split - 1) * -(-chunks // split) + (chunks - 1) // split + 1) * parts * 8192
                        assert traded >= (last if split > 1 else 0) and traded <= stages * stage
                        assert smem == stages * stage + 1024 <= 226 * 1024 // per_sm
                        # (no more CTAs on an SM than it has TMEM columns for)
                        assert (per_sm + 1) * (smem + 1024) > 228 * 1024
    for bad in ((0, 0, 8, 8), (0, 513, 8192, 8192), (0, 1, 0, 8), (0, 1, 8, 12), (3, 1, 8, 8), (-1, 1, 8, 8)):
        assert lib.decoder_gemm_plan(*bad, 152, out) != 0
