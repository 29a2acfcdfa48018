"""Templates and strain far from one: scaled by powers of two, which FP32
arithmetic carries exactly, a search gives the scaled results of the unscaled
one as long as the spectra themselves stay inside the FP32 range, in every
form.  2^104 times 16 to 65536 unit-variance samples leaves spectra of at most
2^114; the inner values of a transform must not leave the range either."""
import numpy as np
import pytest

import synthetic as S
from gpu_helpers import make_ctx

pytestmark = pytest.mark.gpu

KAPPA = 3.0
ROWS = 40
# rows of every size next to one another against strain scaled down, and the
# other way (2^-90: the smallest products stay above FP32's smallest number)
UP, DOWN = np.array([104, 60, 100, 30, 104, 104, 95, 10] * 5), np.full(ROWS, -90)


@pytest.fixture(scope="module")
def ctx():
    c = make_ctx(tail_capacity=1 << 16)
    yield c
    c.close()


def _inputs(n, length):
    bank = S.random_samples_bank(ROWS, length, n + length).astype(np.float32)
    return S.band_limited_noise(n, 3).astype(np.float32), bank


def _scaled(y, bank, strain, rows):
    return np.ldexp(y, strain).astype(np.float32), np.ldexp(bank, rows[:, None]).astype(np.float32)


def _search(ctx, y, bank):
    seg, bid = ctx.bege_load_segment(y), ctx.bege_define_bank_samples(bank)
    dump = ctx.bege_dump_correlation(seg, bid, 0, ROWS)
    job = ctx.bege_correlate(seg, bid, 0, ROWS, KAPPA)
    recs, total = ctx.bege_fetch_tails(job, sort=True)
    assert total == len(recs)
    sigma = ctx.bege_get_sigma(job, ROWS)
    ctx.bege_release(job)
    return seg, bid, dump, recs.copy(), sigma


def _same(dump, recs, sigma, ref, strain, rows):
    # equal but for the rounding of values that reach FP32's subnormal numbers,
    # 2^-23 of the others at most
    want_dump, want, want_sigma = ref
    e = strain + rows
    assert np.isfinite(sigma).all()
    assert np.allclose(np.ldexp(sigma.astype(np.float64), -e), want_sigma, rtol=1e-6, atol=0)
    assert np.array_equal(recs["tmpl"], want["tmpl"]) and np.array_equal(recs["lag"], want["lag"])
    assert np.allclose(np.ldexp(recs["value"].astype(np.float64), -e[recs["tmpl"]]), want["value"],
                       rtol=1e-6, atol=0)
    if dump is not None:
        err = np.abs(np.ldexp(dump.astype(np.float64), -e[:, None]) - want_dump).max(axis=1)
        assert (err <= 1e-6 * want_sigma).all()


def _projection(ctx, y, bank, n):
    seg, bid = ctx.bege_load_segment(y), ctx.bege_define_bank_samples(bank)
    job = ctx.bege_correlate_ex(seg, bid, 0, ROWS, KAPPA, kappa_hi=5.0, linear=True, project=True)
    recs, _ = ctx.bege_fetch_tails(job, sort=True)
    out = recs[["tmpl", "lag"]].tolist(), *ctx.bege_fetch_max(job, n)
    for h in (job, seg, bid):
        ctx.bege_release(h)
    return out


SIZES = [(1 << 10, 1 << 10), (1 << 10, 300), (1 << 11, 300), (1 << 12, 4096), (1 << 13, 4096),
         (1 << 14, 4096), (1 << 14, 1 << 14), (1 << 15, 4096), (1 << 15, 8193), (1 << 16, 4096),
         (1 << 16, 9000), (1 << 17, 4096), (1 << 17, 40000)]


@pytest.mark.parametrize("strain,rows", [(-70, UP), (104, DOWN)], ids=["rows_up", "strain_up"])
@pytest.mark.parametrize("n,length", SIZES)
def test_single_search_in_every_shape(ctx, n, length, strain, rows):
    y, bank = _inputs(n, length)
    handles = _search(ctx, y, bank)
    ref = handles[2:]
    default = ctx.bege_get_config(n)
    for shape in ctx.bege_list_configs(n):
        ctx.bege_set_config(n, *shape)
        seg, bid, *got = _search(ctx, *_scaled(y, bank, strain, rows))
        _same(*got, ref, strain, rows)
        handles += (seg, bid)
    ctx.bege_set_config(n, *default)
    for h in handles[:2] + handles[5:]:
        ctx.bege_release(h)
    want = _projection(ctx, y, bank, n)
    got = _projection(ctx, *_scaled(y, bank, strain, rows), n)
    assert got[0] == want[0] and np.array_equal(got[2], want[2])
    assert np.allclose(got[1], want[1], rtol=1e-6, atol=0)


@pytest.mark.parametrize("strain,rows", [(-70, UP), (104, DOWN)], ids=["rows_up", "strain_up"])
@pytest.mark.parametrize("lg", [14, 15, 16, 17])
def test_block_and_batch(ctx, lg, strain, rows):
    n, length = 1 << lg, 4096
    y, bank = _inputs(n, length)
    h0, b0, *ref = _search(ctx, y, bank)
    ys, banks = _scaled(y, bank, strain, rows)
    seg, bid, dump, recs, sigma = _search(ctx, ys, banks)
    _same(dump, recs, sigma, ref, strain, rows)
    for job in ctx.bege_correlate_multi([seg, seg, seg], bid, 0, ROWS, KAPPA):
        got, _ = ctx.bege_fetch_tails(job, sort=True)
        assert np.array_equal(got, recs)
        assert np.array_equal(ctx.bege_get_sigma(job, ROWS), sigma)
        ctx.bege_release(job)
    batch = ctx.bege_batch_create([(ys, bid, 0, ROWS, KAPPA)])
    for plan in (0, 1):
        ctx.bege_batch_set_plan(batch, plan, 7)
        ctx.bege_batch_run(batch)
        got, _ = ctx.bege_batch_fetch_tails(batch, 0)
        assert np.array_equal(got[np.lexsort((got["lag"], got["tmpl"]))], recs)
        assert np.array_equal(ctx.bege_batch_get_sigma(batch, 0, ROWS), sigma)
    for h in (batch, seg, bid, h0, b0):
        ctx.bege_release(h)


@pytest.mark.parametrize("strain,rows", [(-70, UP), (104, DOWN)], ids=["rows_up", "strain_up"])
@pytest.mark.parametrize("n,length", [(1 << 10, 304), (1 << 13, 4096), (1 << 15, 4096),
                                      (1 << 16, 9000)])
def test_search_without_allocation(ctx, n, length, strain, rows):
    torch = pytest.importorskip("torch")
    from paper_1708_01609_gb300 import binding
    y, bank = _inputs(n, length)
    ys, banks = _scaled(y, bank, strain, rows)
    seg, bid, _, want, want_sigma = _search(ctx, ys, banks)
    dy, db = torch.from_numpy(ys).cuda(), torch.from_numpy(banks).cuda()
    sigma = torch.empty(ROWS, device="cuda")
    recs = torch.empty(1 << 16, 3, dtype=torch.int32, device="cuda")
    total = torch.zeros(1, dtype=torch.int64, device="cuda")
    for _ in range(2):                             # the second call starts its count anew
        binding.bege_search_noalloc(dy.data_ptr(), n, db.data_ptr(), length, 0, ROWS, KAPPA,
                                    sigma.data_ptr(), recs.data_ptr(), len(recs),
                                    total.data_ptr(), torch.cuda.current_stream().cuda_stream)
    got = recs[:int(total.item())].cpu().numpy().reshape(-1).view(binding.TAIL_DTYPE)
    assert np.array_equal(got[np.lexsort((got["lag"], got["tmpl"]))], want)
    assert np.array_equal(sigma.cpu().numpy(), want_sigma)
    ctx.bege_release(seg)
    ctx.bege_release(bid)


def test_values_that_are_not_finite_stay_so(ctx):
    """Rows with an infinity or a NaN, or a correlation beyond FP32, have no
    finite sigma and no tails; their neighbours are as ever."""
    for n in (1 << 10, 1 << 14, 1 << 16):
        y, bank = _inputs(n, 1000)
        ref = _search(ctx, y, bank)
        bad = bank.copy()
        bad[3, 5], bad[10, 0], bad[11] = np.inf, np.nan, bad[11] * np.float32(1e25)
        bad[12, 7] = np.float32(3e38)
        seg, bid, _, recs, sigma = _search(ctx, y, bad)
        rest = np.setdiff1d(np.arange(ROWS), [3, 10, 11, 12])
        assert not np.isfinite(sigma[[3, 10, 11, 12]]).any()
        assert np.isin(recs["tmpl"], rest).all()
        assert np.array_equal(sigma[rest], ref[4][rest])
        assert np.array_equal(recs, ref[3][np.isin(ref[3]["tmpl"], rest)])
        for h in (seg, bid, *ref[:2]):
            ctx.bege_release(h)
