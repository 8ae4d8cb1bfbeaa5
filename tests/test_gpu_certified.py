"""Searches through the certified tensor-core filter (many queries per probed
list) give the direct scans' ids and distance bits: the re-score uses the
scan's arithmetic, and the filter keeps every member that can be among the k
nearest, so no tolerance applies."""
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


def make(P, n, d, nlist, B, seed, d_c=16):
    data = synthdata.small(n, B, d, 24, seed)
    db = torch.from_numpy(data["db"]).cuda()
    g = P.build_ivf(db, d_c, nlist, 4, n, seed)
    return data, g, torch.from_numpy(data["queries"]).cuda()


def both(P, g, q, *args, filtered=True):
    """(filtered, tiled): the option that turns the streaming scan off keeps the tiled scan."""
    P.profile_enable(True)
    a = [t.cpu().numpy() for t in P.search_ivf(g, q, *args, return_probes=True)]
    assert ("mma" in P.profile_read()) == filtered
    P.profile_enable(False)
    with P.option(P.OPT_FP32_STREAM, 0):
        b = [t.cpu().numpy() for t in P.search_ivf(g, q, *args, return_probes=True)]
    g.status()
    return a, b


def same(a, b):
    for x, y in zip(a, b):
        np.testing.assert_array_equal(x.view(np.int32) if x.dtype == np.float32 else x,
                                      y.view(np.int32) if y.dtype == np.float32 else y)


# d_s across the 64-coordinate blocks (remainders 8, 16, 32, 48), k from 1 to
# the largest the filter takes and one above, few and many probes
@pytest.mark.parametrize("d,d_s,nprobe,k,B", [
    (64, 8, 4, 10, 4003), (64, 48, 4, 1, 700), (64, 64, 24, 100, 333), (96, 96, 3, 7, 3000),
    (256, 192, 9, 100, 1500), (256, 256, 12, 256, 900), (256, 256, 12, 257, 300),
    (512, 512, 5, 33, 5000), (1024, 1024, 6, 100, 1100)])
def test_equals_tiled_scan(P, d, d_s, nprobe, k, B):
    _, g, q = make(P, 6000, d, 24, B, d_s + k)
    same(*both(P, g, q, 16, d_s, nprobe, k, filtered=k <= 256))
    g.free()


def test_left_over_queries(P):
    """Queries whose certified set overflows (zero queries, exact duplicates of
    hundreds of rows) share a batch with ordinary ones."""
    data = synthdata.small(5000, 900, 64, 16, 5)
    db, q = data["db"].copy(), data["queries"].copy()
    db[1000:2500] = db[7]          # 1,500 equal rows
    db[3000:3040] = 0              # zero vectors
    q[::7] = 0
    q[3::11] = db[7]
    db, q = torch.from_numpy(db).cuda(), torch.from_numpy(q).cuda()
    g = P.build_ivf(db, 16, 12, 4, 5000, 3)
    a, b = both(P, g, q, 16, 64, 6, 50)
    same(a, b)
    g.free()


def test_empty_lists_and_few_candidates(P):
    """Lists of 0 to 300 members, some queries with fewer than k candidates."""
    data = synthdata.small(1500, 1500, 64, 16, 9)
    rng = np.random.default_rng(1)
    assign = rng.choice([0, 2, 3, 5, 7], size=1500, p=[.2, .3, .3, .19, .01]).astype(np.int32)
    cent = torch.from_numpy(data["means"][:10, :16].copy()).cuda()
    g = P.index_create(torch.from_numpy(data["db"]).cuda(), cent, torch.from_numpy(assign).cuda())
    same(*both(P, g, torch.from_numpy(data["queries"]).cuda(), 16, 64, 2, 60))
    g.free()


def test_tiny_and_huge_magnitudes(P):
    """Rows and queries whose squared norms leave FP32's normal range."""
    data = synthdata.small(3000, 600, 64, 16, 21)
    db, q = data["db"].copy(), data["queries"].copy()
    db[::5] *= 1e-22
    db[1::5] *= 1e18
    q[::3] *= 1e-22
    db, q = torch.from_numpy(db).cuda(), torch.from_numpy(q).cuda()
    g = P.build_ivf(db, 16, 12, 3, 3000, 3)
    same(*both(P, g, q, 16, 64, 4, 20))
    g.free()


def test_slices(P):
    """A scratch budget that cuts the batch into slices."""
    _, g, q = make(P, 20000, 128, 16, 4000, 77)
    with P.option(P.OPT_SCRATCH_BYTES, 48 << 20):
        a, b = both(P, g, q, 16, 128, 4, 40)
    same(a, b)
    same(a, both(P, g, q, 16, 128, 4, 40)[0])
    g.free()


# ------------------------------------------------------------------ IVF-OPQ
def opq_index(P, n, d, d_s, M, nlist, seed, db=None):
    """An index with a random orthonormal rotation and codebooks of sampled rows."""
    data = synthdata.small(n, 8, d, 24, seed)
    x = torch.from_numpy(data["db"] if db is None else db).cuda()
    g = P.build_ivf(x, 16, nlist, 3, n, seed) if nlist > 1 else P.flat_index(x)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    R = torch.linalg.qr(torch.randn(d_s, d_s, device="cuda", generator=gen))[0].contiguous()
    z = torch.nn.functional.normalize(x[:256, :d_s], dim=1) @ R
    C = z.view(256, M, d_s // M).transpose(0, 1).contiguous()
    P.set_opq(g, d_s, M, R, C, P.opq_encode(x, d_s, M, R, C))
    return data["means"], g


def opq_both(P, g, q, *args, filtered=True, **kw):
    """(filtered, lookups): the option that turns distance-then-select off keeps
    the running top-k over table lookups."""
    P.profile_enable(True)
    a = [t.cpu().numpy() for t in P.search_ivfopq(g, q, *args, return_probes=True, **kw)]
    # the cluster mapping has no stage of that name
    assert ("mma" in P.profile_read()) == filtered
    P.profile_enable(False)
    with P.option(P.OPT_ADC_SELECT, 0):
        b = [t.cpu().numpy() for t in P.search_ivfopq(g, q, *args, return_probes=True, **kw)]
    g.status()
    return a, b


# sub-vectors of 1 to 16 coordinates (whole and crossing groups of four),
# sums of words and of bytes, one list and several, shortlists up to the
# largest filtered one and one above
@pytest.mark.parametrize("d,d_s,M,nlist,nprobe,k,rerank,B", [
    (64, 64, 8, 4, 4, 10, 0, 3601), (64, 64, 64, 4, 3, 100, 400, 700),
    (96, 96, 32, 4, 4, 5, 0, 1000), (96, 96, 6, 1, 1, 10, 0, 8001),
    (128, 128, 16, 1, 1, 10, 40, 2047), (256, 192, 16, 6, 5, 100, 0, 2500),
    (384, 384, 32, 6, 6, 128, 512, 800), (384, 384, 32, 6, 6, 128, 513, 800)])
def test_opq_equals_lookups(P, d, d_s, M, nlist, nprobe, k, rerank, B):
    means, g = opq_index(P, 20000, d, d_s, M, nlist, d_s + M)
    q = torch.from_numpy(synthdata.sample_points(B, d, means, 99, threads=1)[0]).cuda()
    same(*opq_both(P, g, q, 8 if nlist == 1 else 16, nprobe, k, rerank_k=rerank,
                   filtered=rerank <= 512))
    g.free()


def test_opq_left_over_queries(P):
    """Thousands of rows with one code: certified sets that overflow, and a
    batch cut into slices by the scratch budget."""
    data = synthdata.small(20000, 8, 64, 16, 31)
    db = data["db"].copy()
    db[2000:6000] = db[5]
    means, g = opq_index(P, 20000, 64, 64, 16, 3, 31, db=db)
    q = synthdata.sample_points(3000, 64, means, 7, threads=1)[0]
    q[::9] = db[5]
    q[4::50] = 0
    q = torch.from_numpy(q).cuda()
    a, b = opq_both(P, g, q, 16, 3, 20, rerank_k=80)
    same(a, b)
    with P.option(P.OPT_SCRATCH_BYTES, 160 << 20):
        c = [t.cpu().numpy() for t in P.search_ivfopq(g, q, 16, 3, 20, rerank_k=80,
                                                      return_probes=True)]
    same(c, b)
    g.free()
