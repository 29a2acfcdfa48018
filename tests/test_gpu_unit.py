"""The correlate kernels at the edges of their range: every segment length,
fewer templates than a CTA has units (N <= 2^13), template lengths around the column length (one sample, odd, half a column, a column, folded
over several), every launch shape, against the FP64 oracle; all shapes give
the same bits, and a row gives the same bits wherever its range begins."""
import numpy as np
import pytest

import synthetic as S
from gpu_helpers import make_ctx, oracle_rho

pytestmark = pytest.mark.gpu

TOL = 1e-5        # sigma; FP32 rounding of the transforms reaches 2e-6


@pytest.fixture(scope="module")
def ctx():
    c = make_ctx()
    yield c
    c.close()


@pytest.mark.parametrize("n,length", [(1 << 10, 1), (1 << 10, 1 << 10), (1 << 11, 513),
                                      (1 << 12, 2049), (1 << 12, 1 << 12), (1 << 13, 4095),
                                      (1 << 13, 4097), (1 << 14, 1), (1 << 14, 4096), (1 << 14, 4097),
                                      (1 << 14, 1 << 14), (1 << 15, 2047), (1 << 15, 8193),
                                      (1 << 16, 7), (1 << 16, 4095), (1 << 16, 1 << 16),
                                      (1 << 17, 4096), (1 << 17, 12289)])
def test_edges_match_oracle_in_every_shape(ctx, n, length):
    bank = S.random_samples_bank(5, length, 3 * n + length)
    bank[3] = 0.0                                  # a row of zeros: no value, no tail
    y = S.band_limited_noise(n, length)
    rho, sig = oracle_rho(y, bank)
    seg, bid = ctx.bege_load_segment(y), ctx.bege_define_bank_samples(bank)
    default = ctx.bege_get_config(n)
    seen = []
    for shape in ctx.bege_list_configs(n):
        ctx.bege_set_config(n, *shape)
        dump = ctx.bege_dump_correlation(seg, bid, 0, 5)
        job = ctx.bege_correlate(seg, bid, 0, 5, 3.0)
        recs, total = ctx.bege_fetch_tails(job, sort=True)
        gsig = ctx.bege_get_sigma(job, 5)
        assert total == len(recs)
        ctx.bege_release(job)
        for k in range(5):
            if k == 3:
                assert gsig[k] == 0 and not dump[k].any() and not (recs["tmpl"] == k).any()
                continue
            assert abs(gsig[k] / sig[k] - 1) <= 1e-6
            assert np.abs(dump[k] - rho[k]).max() <= TOL * sig[k]
            hits = np.nonzero(np.abs(dump[k]) > np.float32(3.0) * gsig[k])[0]
            mine = recs[recs["tmpl"] == k]
            assert np.array_equal(mine["lag"], hits)
            assert np.array_equal(mine["value"], dump[k][hits])
        # the same row from a range that begins elsewhere
        job = ctx.bege_correlate(seg, bid, 4, 5, 3.0)
        assert ctx.bege_get_sigma(job, 1)[0] == gsig[4]
        ctx.bege_release(job)
        seen.append((dump, gsig, recs.copy()))
    ctx.bege_set_config(n, *default)
    for other in seen[1:]:
        for a, b in zip(seen[0], other):
            assert np.array_equal(a, b)
    ctx.bege_release(seg)
    ctx.bege_release(bid)


def test_coefficients_and_tables_at_a_quarter_turn(ctx):
    """One bin at a time: a cosine at bin j against a unit impulse gives the
    cosine back at every lag (twiddles at 0, 1/4 and 1/2 turn, the self-mirrored
    butterflies and both ends of the spectrum included)."""
    n = 1 << 16
    bank = np.zeros((1, 8), dtype=np.float32)
    bank[0, 0] = 1.0
    bid = ctx.bege_define_bank_samples(bank)
    t = np.arange(n)
    for j in (0, 1, 8, 128, 2048, 4096, 8192, 16383, 16384, 16385, 24576, 32767, 32768):
        y = np.cos(2 * np.pi * ((j * t) % n) / n).astype(np.float32)
        seg = ctx.bege_load_segment(y)
        dump = ctx.bege_dump_correlation(seg, bid, 0, 1)[0]
        ctx.bege_release(seg)
        assert np.abs(dump - y).max() <= 2e-6, j
    ctx.bege_release(bid)


@pytest.mark.parametrize("n,length", [(1 << 16, 4096), (1 << 17, 4096), (1 << 17, 5000)])
def test_exchange_through_l2_equals_shared_memory(ctx, n, length):
    """N >= 2^16 exchanges columns through a buffer one template behind; a
    context with a budget does without it.  Same bits, over several templates
    per cluster and a last round that not every cluster takes part in, in both
    epilogues."""
    count = 401
    bank = S.random_samples_bank(count, length, n + length)
    y = S.band_limited_noise(n, 5)
    got, extended = [], []
    small = make_ctx(hbm_budget_bytes=1 << 30)
    for c in (ctx, small):
        seg, bid = c.bege_load_segment(y), c.bege_define_bank_samples(bank)
        c.bege_set_config(n, 4, 512)
        for k0, k1 in ((0, count), (7, 8)):
            job = c.bege_correlate(seg, bid, k0, k1, 3.5)
            recs, total = c.bege_fetch_tails(job, sort=True)
            assert total == len(recs) > 0
            got.append((recs.copy(), c.bege_get_sigma(job, k1 - k0)))
            c.bege_release(job)
        job = c.bege_correlate_ex(seg, bid, 0, count, 3.5, kappa_hi=4.5, linear=True, project=True)
        recs, total = c.bege_fetch_tails(job, sort=True)
        assert total == len(recs) > 0
        extended.append((recs.copy(), *c.bege_fetch_max(job, n)))
        c.bege_release(job)
        c.bege_release(seg)
        c.bege_release(bid)
    small.close()
    for a, b in zip(got[:2], got[2:]):
        assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
    for a, b in zip(*extended):
        assert np.array_equal(a, b)
    all_, one = got[0], got[1]
    assert one[1][0] == all_[1][7]
    assert np.array_equal(one[0], all_[0][all_[0]["tmpl"] == 7])


@pytest.mark.parametrize("lg", [10, 11, 12, 13, 14])
def test_rounds_of_the_short_kernels(ctx, lg):
    """More templates than the GPU holds at once: rows of the first round, the
    second and a last one that ends within a CTA, against the oracle, and the
    same bits as a search of that row alone."""
    torch = pytest.importorskip("torch")
    n, length = 1 << lg, 300
    units = 2 * torch.cuda.get_device_properties(0).multi_processor_count * (1 << (14 - lg))
    count = 2 * units + 3
    bank = S.random_samples_bank(count, length, lg)
    y = S.band_limited_noise(n, 9)
    seg, bid = ctx.bege_load_segment(y), ctx.bege_define_bank_samples(bank)
    job = ctx.bege_correlate(seg, bid, 0, count, 4.0)
    recs, total = ctx.bege_fetch_tails(job, sort=True)
    assert total == len(recs)
    sigma = ctx.bege_get_sigma(job, count)
    ctx.bege_release(job)
    rows = [0, 1, units - 1, units, units + 17, 2 * units - 1, 2 * units, count - 2, count - 1]
    _, want = oracle_rho(y, bank[rows])
    for k, ref in zip(rows, want):
        assert abs(sigma[k] / ref - 1) <= 1e-6
        job = ctx.bege_correlate(seg, bid, k, k + 1, 4.0)
        one, _ = ctx.bege_fetch_tails(job, sort=True)
        assert ctx.bege_get_sigma(job, 1)[0] == sigma[k]
        assert np.array_equal(one, recs[recs["tmpl"] == k])
        ctx.bege_release(job)
    ctx.bege_release(seg)
    ctx.bege_release(bid)
