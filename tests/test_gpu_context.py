"""What a context keeps between calls."""
import numpy as np
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


@pytest.mark.parametrize("idle_buffer", [False, True])
def test_capture_of_a_search_allocates_nothing(idle_buffer):
    """A search enqueued on a stream under capture takes no exchange buffer,
    new or idle, and leaves the capture valid; the graph runs, and later
    searches are as ever."""
    torch = pytest.importorskip("torch")
    n = 1 << 16
    with make_ctx(tail_capacity=1 << 12) as ctx:
        bank = ctx.bege_define_bank_samples(S.random_samples_bank(20, 64, 1))
        seg = ctx.bege_load_segment(S.band_limited_noise(n, 1))
        if not idle_buffer:
            ctx.bege_set_config(n, 2, 256)      # this shape has no use for one
        job = ctx.bege_correlate(seg, bank, 0, 20, 5.0)
        want = ctx.bege_get_sigma(job, 20)
        ctx.bege_release(job)
        ctx.bege_set_config(n, 4, 512)
        held = ctx.bege_device_bytes()
        graph, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
        with torch.cuda.graph(graph, stream=stream):
            job = ctx.bege_correlate(seg, bank, 0, 20, 5.0, stream.cuda_stream)
        assert ctx.bege_device_bytes() == held
        for _ in range(2):
            graph.replay()
        torch.cuda.synchronize()
        second = ctx.bege_correlate(seg, bank, 0, 20, 5.0)
        assert np.array_equal(ctx.bege_get_sigma(second, 20), want)
        del graph
        for h in (second, job, seg, bank):
            ctx.bege_release(h)


def test_job_time_is_the_kernel_alone():
    """The first job of a context, whose buffers are allocated in the call,
    reports the time of its kernel as later ones do."""
    n = 1 << 16
    bank_rows = S.random_samples_bank(300, 64, 1)
    y = S.band_limited_noise(n, 3)
    first, later = [], []
    for _ in range(5):
        with make_ctx(tail_capacity=1 << 12) as ctx:
            bank = ctx.bege_define_bank_samples(bank_rows)
            seg = ctx.bege_load_segment(y)
            for times in (first, later, later):
                job = ctx.bege_correlate(seg, bank, 0, 300, 5.0)
                times.append(ctx.bege_job_kernel_ms(job))
                ctx.bege_release(job)
    assert min(first) <= 1.3 * np.median(later), (first, later)


def test_kept_buffers_are_bounded_and_give_way():
    """Released segments leave at most 4 MB behind, and none of it stands in the
    way of an allocation that the budget allows."""
    n = 1 << 16
    segment = 8 * (n // 2 + 1) + 16 * (n // 2)
    with make_ctx(tail_capacity=1 << 12, hbm_budget_bytes=32 << 20) as ctx:
        segs = [ctx.bege_load_segment(S.band_limited_noise(n, i)) for i in range(12)]
        used = ctx.bege_device_bytes()
        for seg in segs:
            ctx.bege_release(seg)
        idle = ctx.bege_device_bytes()
        assert used - 12 * segment <= idle <= used - 12 * segment + (4 << 20)
        tables = idle - (4 << 20)                  # at most: the plan of n stays
        rows = ((32 << 20) - tables - (1 << 20)) // (4096 * 4)
        bank = ctx.bege_define_bank_samples(np.zeros((rows, 4096), np.float32))
        assert idle + rows * 4096 * 4 > 32 << 20   # fits only without the kept buffers
        ctx.bege_release(bank)


def test_segment_buffers_are_reused_after_their_jobs():
    """A segment released while its search runs on one stream, and the next one
    of that length loaded on another, which takes its buffers."""
    torch = pytest.importorskip("torch")
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    for n, count in ((1 << 13, 40000), (1 << 15, 20000)):
        length = 4096
        params = np.stack([np.linspace(400.0, 1500.0, count), np.zeros(count)], axis=1)
        y = [S.band_limited_noise(n, i) for i in (1, 2)]
        with make_ctx(tail_capacity=1 << 16) as ctx:
            bank = ctx.bege_define_bank(params, tau=length / 4096.0)
            want = []
            for strain in y:
                seg = ctx.bege_load_segment(strain)
                job = ctx.bege_correlate(seg, bank, 0, count, 5.0)
                want.append(ctx.bege_get_sigma(job, count))
                ctx.bege_release(job)
                ctx.bege_release(seg)
            seg = ctx.bege_load_segment(y[0], 0, a.cuda_stream)
            first = ctx.bege_correlate(seg, bank, 0, count, 5.0, a.cuda_stream)
            ctx.bege_release(seg)
            seg = ctx.bege_load_segment(y[1], 0, b.cuda_stream)
            second = ctx.bege_correlate(seg, bank, 0, count, 5.0, b.cuda_stream)
            assert np.array_equal(ctx.bege_get_sigma(first, count), want[0])
            assert np.array_equal(ctx.bege_get_sigma(second, count), want[1])
