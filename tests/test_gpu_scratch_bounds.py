"""The documented bound of a search's scratch (what the server admits batches by)
holds for every route, nested steps included, and a filtered call stays within the
scratch budget it was given."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import paper_2305_19435_gb300 as P
    P.build()
    assert torch.cuda.is_available()
    return P


def make(P, N, d, nlist, **kw):
    """Rows and centroids at random, lists of equal length but for a longer first one."""
    gen = torch.Generator(device="cuda").manual_seed(N + d)
    db = torch.randn(N, d, device="cuda", generator=gen)
    assign = torch.arange(N, device="cuda", dtype=torch.int32) % nlist
    assign[N - N // 50:] = 0
    cent = torch.nn.functional.normalize(torch.randn(nlist, 16, device="cuda", generator=gen))
    return P.index_create(db, cent, assign, **kw), torch.randn(50000, d, device="cuda", generator=gen)


def held(P, f):
    torch.cuda.synchronize()
    P.scratch_high(reset=True)
    f()
    return P.scratch_high()


# (B, d_s, probes, k): the filter with a large cluster mapping, the streaming scan with
# and without its unit table, the tiled scan (k 1), one query
@pytest.mark.parametrize("metric", [0, 1])
def test_fp32(P, metric):
    g, q = make(P, 60000, 64, 1024, metric=metric)
    for B, d_s, npb, k in [(50000, 64, 4, 10), (50000, 16, 1, 1), (3000, 64, 8, 100), (500, 64, 16, 10),
                           (1, 8, 16, 1000), (64, 64, 128, 1024), (40, 64, 300, 10)]:
        n = held(P, lambda: P.search_ivf(g, q[:B], 16, d_s, npb, k))
        assert 0 < n <= P.scratch_bytes(g, B, 16, d_s, npb, k), (B, d_s, npb, k)
    with P.option(P.OPT_FP32_STREAM, 0):
        n = held(P, lambda: P.search_ivf(g, q, 16, 64, 4, 100))
        assert 0 < n <= P.scratch_bytes(g, 50000, 16, 64, 4, 100)
    g.free()


def test_low_precision_and_padding(P):
    """256 lists of long rows: a part-filled query tile per list is most of it."""
    g, q = make(P, 20000, 2048, 256, storage=P.STORE_F32 | P.STORE_BF16 | P.STORE_FP8)
    calls = [(P.STORE_F32, 4000, 2048, 8, 100, 0), (P.STORE_F32, 600, 2048, 4, 10, 0)]
    for tier in (P.STORE_BF16, P.STORE_FP8):  # wide and narrow tiles, both reranks
        calls += [(tier, 4000, 2048, 8, 10, 40), (tier, 600, 2048, 4, 10, 40),
                  (tier, 20000, 64, 4, 100, 400), (tier, 1, 512, 16, 10, 10)]
    for tier, B, d_s, npb, k, rr in calls:
        f = lambda: P.search_ivf(g, q[:B], 16, d_s, npb, k, storage=tier, rerank_k=rr)
        assert 0 < held(P, f) <= P.scratch_bytes(g, B, 16, d_s, npb, k, tier, rr), (tier, B, d_s)
        if tier != P.STORE_F32:
            with P.option(P.OPT_SCAN_FILTER, 1):
                assert 0 < held(P, f) <= P.scratch_bytes(g, B, 16, d_s, npb, k, tier, rr)
    # slices of a filtered batch, and no filter where its padding leaves no room
    for budget in (800 << 20, 300 << 20, 100 << 20):
        with P.option(P.OPT_SCRATCH_BYTES, budget):
            f = lambda: P.search_ivf(g, q[:8000], 16, 2048, 8, 100)
            n = held(P, f)
            assert 0 < n <= P.scratch_bytes(g, 8000, 16, 2048, 8, 100)
            assert n <= budget + (16 << 20) or budget < 800 << 20
    g.free()


def test_ivfopq(P):
    """The lookup scan, the filter (whose FP16 rows count, at more than one part of the
    batch too) and the running top-k scan; both servers admit by the same bound."""
    from paper_2305_19435_gb300.serving import Budget, GpuExecutor
    g, q = make(P, 60000, 128, 256)
    R, C = torch.eye(128, device="cuda"), 0.05 * torch.randn(32, 256, 4, device="cuda")
    codes = torch.randint(0, 256, (60000, 32), device="cuda", dtype=torch.uint8)
    assert P.ivfopq_scratch_bytes(g, 10, 16, 4, 10) == -1  # no codes yet
    P.set_opq(g, 128, 32, R, C, codes)
    ex = GpuExecutor({0: g}, 1)
    for B, npb, k, rr, filtered in [(8000, 16, 10, 0, True), (8000, 16, 100, 400, True),
                                    (200, 16, 10, 40, False), (1, 4, 10, 0, False),
                                    (8000, 1, 100, 1000, False), (300, 256, 10, 100, False)]:
        for budget in (12 << 30, 400 << 20):
            with P.option(P.OPT_SCRATCH_BYTES, budget):
                bound = P.ivfopq_scratch_bytes(g, B, 16, npb, k, rr)
                P.profile_enable(True)
                n = held(P, lambda: P.search_ivfopq(g, q[:B], 16, npb, k, rerank_k=rr))
                assert ("mma" in P.profile_read()) == filtered
                P.profile_enable(False)
                assert 0 < n <= bound, (B, npb, k, rr)
                assert ex.scratch_bytes(0, Budget(16, 128, npb, k, 0, rr, 1), B) == bound
                assert not filtered or bound >= 60000 * 2 * 128
                assert n <= budget + (16 << 20) or B == 8000 and not filtered
    with P.option(P.OPT_ADC_SELECT, 0):
        for B, npb, k, rr in [(8000, 16, 10, 0), (3000, 16, 100, 400), (1, 300 - 44, 10, 10)]:
            n = held(P, lambda: P.search_ivfopq(g, q[:B], 16, npb, k, rerank_k=rr))
            assert 0 < n <= P.ivfopq_scratch_bytes(g, B, 16, npb, k, rr), (B, npb, k, rr)
    g.free()
