"""What a context keeps between calls."""
import pytest

import synthetic as S
from gpu_helpers import make_ctx

pytestmark = pytest.mark.gpu


def test_sequential_searches_share_one_exchange_buffer():
    """However many job buffers earlier calls left behind, searches that run
    one after the other hold one exchange buffer (at most 40 MB) between them."""
    n = 1 << 16
    with make_ctx(tail_capacity=1 << 12) as ctx:
        bank = ctx.bege_define_bank_samples(S.random_samples_bank(300, 64, 1))
        segs = [ctx.bege_load_segment(S.band_limited_noise(n, i)) for i in range(8)]
        for j in ctx.bege_correlate_multi(segs, bank, 0, 300, 5.0):
            ctx.bege_release(j)
        before = ctx.bege_device_bytes()
        held = []
        for i in range(8):
            job = ctx.bege_correlate(segs[i], bank, 0, 300, 5.0)
            ctx.bege_get_sigma(job, 300)
            ctx.bege_release(job)
            held.append(ctx.bege_device_bytes() - before)
        assert 0 < held[0] <= 40 << 20
        assert held == held[:1] * 8
