"""Searches that cannot have the scratch of their fastest route take one that
needs less, with the same ids and distance bits; a limit on the library's
scratch (a test hook) stands in for a device without free memory."""
import numpy as np
import pytest

import synthdata

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import paper_2305_19435_gb300 as P
    P.build()
    assert torch.cuda.is_available()
    return P


@pytest.fixture(scope="module")
def data():
    return synthdata.small(20000, 4000, 128, 24, 77)


def same(a, b):
    for x, y in zip(a, b):
        x, y = x.cpu().numpy(), y.cpu().numpy()
        np.testing.assert_array_equal(x.view(np.int32) if x.dtype == np.float32 else x,
                                      y.view(np.int32) if y.dtype == np.float32 else y)


def profiled(P, f):
    P.profile_enable(True)
    r = f()
    stages = P.profile_read()
    P.profile_enable(False)
    return r, stages


# the filter's keys alone are 52 MB at least, the tiled scan's partial results a
# few; the raw metric has no filter (streaming scan: 4 bytes per probed member)
@pytest.mark.parametrize("metric,B", [("prefixnorm", 4000), ("l2", 2000)])
def test_fp32_falls_back(P, data, metric, B):
    db, q = torch.from_numpy(data["db"]).cuda(), torch.from_numpy(data["queries"][:B]).cuda()
    m = P.METRIC_L2 if metric == "l2" else P.METRIC_L2_PREFIXNORM
    g = P.build_ivf(db, 16, 16, 4, 20000, 77, metric=m)
    f = lambda: P.search_ivf(g, q, 16, 128, 4, 10, return_probes=True)
    want, stages = profiled(P, f)
    assert ("mma" in stages) == (metric == "prefixnorm")
    with P.option(P.OPT_TEST_SCRATCH_LIMIT, 24 << 20):
        got, stages = profiled(P, f)
        assert "mma" not in stages and "scan" in stages
        plan = P.Plan(g, q, 16, 128, 4, 10)
    same(got, want)
    want1 = want
    same(plan.launch(), want[:2])
    plan.free()
    rng = np.random.default_rng(B)
    ds, npr = rng.choice([64, 128], B).tolist(), rng.integers(1, 5, B).tolist()
    f = lambda: P.search_ivf_budgets(g, q, 16, ds, npr, [10] * B)
    want = f()
    with P.option(P.OPT_TEST_SCRATCH_LIMIT, 24 << 20):
        got = f()
    same(got, want)
    # not even the tiled scan's: the documented error, and the next call is whole
    with P.option(P.OPT_TEST_SCRATCH_LIMIT, 1 << 20), pytest.raises(P.AdannsError):
        P.search_ivf(g, q, 16, 128, 4, 10)
    same(P.search_ivf(g, q, 16, 128, 4, 10), want1[:2])
    g.status()
    g.free()


def test_ivfopq_falls_back(P, data):
    """The filter's FP16 rows (5 MB) on top of the lookup scan's scratch."""
    db, q = torch.from_numpy(data["db"]).cuda(), torch.from_numpy(data["queries"][:3000]).cuda()
    g = P.flat_index(db)
    R = torch.eye(128, device="cuda")
    z = torch.nn.functional.normalize(db[:256], dim=1)
    C = z.view(256, 16, 8).transpose(0, 1).contiguous()
    P.set_opq(g, 128, 16, R, C, P.opq_encode(db, 128, 16, R, C))
    for kw in ({}, {"rerank_k": 40}):
        f = lambda: P.search_ivfopq(g, q, 8, 1, 10, return_probes=True, **kw)
        want, stages = profiled(P, f)
        assert "mma" in stages
        # MiB: scores 229, tables 47, the rest under 8; the filter 31 more
        with P.option(P.OPT_TEST_SCRATCH_LIMIT, 296 << 20):
            got, stages = profiled(P, f)
        assert "mma" not in stages and "adc" in stages
        same(got, want)
    want = P.search_ivfopq_budgets(g, q, 8, [1] * 3000, [10] * 3000)
    with P.option(P.OPT_TEST_SCRATCH_LIMIT, 296 << 20):
        same(P.search_ivfopq_budgets(g, q, 8, [1] * 3000, [10] * 3000), want)
    g.free()


def test_codes_load_without_their_norms(P, data):
    """The code rows' norms are only for the filter: codes load without them,
    and the lookup scan answers."""
    db, q = torch.from_numpy(data["db"]).cuda(), torch.from_numpy(data["queries"][:3000]).cuda()
    g = P.flat_index(db)
    R = torch.eye(128, device="cuda")
    z = torch.nn.functional.normalize(db[:256], dim=1)
    C = z.view(256, 16, 8).transpose(0, 1).contiguous()
    codes = P.opq_encode(db, 128, 16, R, C)
    f = lambda: P.search_ivfopq(g, q, 8, 1, 10, return_probes=True)
    P.set_opq(g, 128, 16, R, C, codes)
    want, stages = profiled(P, f)
    assert "mma" in stages
    with P.option(P.OPT_TEST_SCRATCH_LIMIT, 0):
        P.set_opq(g, 128, 16, R, C, codes)
    got, stages = profiled(P, f)
    assert "mma" not in stages and "adc" in stages
    same(got, want)
    P.set_opq(g, 128, 16, R, C, codes)
    assert "mma" in profiled(P, f)[1]
    g.free()


def test_residual_codes_hold_no_norms(P):
    """Residual codes are never searched by the filter: loading them takes the
    codes (N M bytes) and the list tables, not 4 bytes per row of code norms."""
    N = 4_000_000
    db = torch.randn(N, 8, device="cuda")
    g = P.flat_index(db)
    R, C = torch.eye(8, device="cuda"), torch.randn(1, 256, 8, device="cuda")
    codes = torch.zeros(N, 1, dtype=torch.uint8, device="cuda")
    centres = torch.zeros(1, 8, device="cuda")

    def held(load):  # by a second load: the pool and the kernels' modules are there
        load()
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        g2 = P.flat_index(db)
        torch.cuda.synchronize()
        bare = before - torch.cuda.mem_get_info()[0]
        load(g2)
        torch.cuda.synchronize()
        used = before - torch.cuda.mem_get_info()[0] - bare
        g2.free()
        return used

    plain = held(lambda x=g: P.set_opq(x, 8, 1, R, C, codes))
    residual = held(lambda x=g: P.set_opq_residual(x, 8, 1, R, C, codes, centres))
    assert plain - residual >= 4 * N - (8 << 20)  # 16 MB; 2 MB pages of the small tables
    g.free()
