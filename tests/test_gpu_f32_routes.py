"""Which route an FP32 batch takes: the certified filter only where it is estimated
to be the fastest.  The results are the tiled scan's, bit for bit, on each."""
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
def index(P):
    data = synthdata.small(20000, 8192, 512, 64, 41)
    g = P.build_ivf(torch.from_numpy(data["db"]).cuda(), 16, 64, 4, 20000, 3)
    yield g, torch.from_numpy(data["queries"]).cuda()
    g.free()


# 256 queries per list: few members per query beside its own cost (k 1 and 10, two
# probes), all of them re-scored (k 256, two probes); enough of them (k 100, eight
# probes); 64 per list at a long and a short prefix
@pytest.mark.parametrize("d_s,nprobe,k,B,filtered", [
    (64, 2, 1, 8192, False), (16, 2, 10, 8192, False), (64, 2, 256, 8192, False),
    (512, 8, 100, 2048, True), (512, 8, 1, 2048, True), (512, 8, 10, 1024, True),
    (16, 8, 1, 512, False)])
def test_route(P, index, d_s, nprobe, k, B, filtered):
    g, q = index
    q = q[:B]
    P.profile_enable(True)
    a = [t.cpu().numpy() for t in P.search_ivf(g, q, 16, d_s, nprobe, k)]
    stages = P.profile_read()
    P.profile_enable(False)
    assert ("mma" in stages) == filtered
    with P.option(P.OPT_FP32_STREAM, 0):
        b = [t.cpu().numpy() for t in P.search_ivf(g, q, 16, d_s, nprobe, k)]
    np.testing.assert_array_equal(a[0], b[0])
    np.testing.assert_array_equal(a[1].view(np.int32), b[1].view(np.int32))


# the raw metric (no filter): at k 1 the tiled scan where the selection's CTA per
# query would be most of the call, told by the scratch of the route
@pytest.mark.parametrize("d_s,nprobe,k,B,tiled", [
    (16, 2, 1, 2880, True), (64, 1, 1, 8192, True), (16, 2, 2, 2880, False),
    (64, 2, 1, 320, False), (16, 2, 1, 500, False)])
def test_stream_or_tiled(P, d_s, nprobe, k, B, tiled):
    data = synthdata.small(20000, 8192, 64, 64, 43)
    g = P.build_ivf(torch.from_numpy(data["db"]).cuda(), 16, 64, 4, 20000, 3, metric=P.METRIC_L2)
    q = torch.from_numpy(data["queries"][:B]).cuda()
    with P.option(P.OPT_FP32_STREAM, 0):
        b = [t.cpu().numpy() for t in P.search_ivf(g, q, 16, d_s, nprobe, k)]
        need = P.scratch_bytes(g, B, 16, d_s, nprobe, k)
    assert (P.scratch_bytes(g, B, 16, d_s, nprobe, k) == need) == tiled
    a = [t.cpu().numpy() for t in P.search_ivf(g, q, 16, d_s, nprobe, k)]
    np.testing.assert_array_equal(a[0], b[0])
    np.testing.assert_array_equal(a[1].view(np.int32), b[1].view(np.int32))
    g.free()


# NaN, infinity, a squared norm that underflows and one that overflows, at the last
# coordinate: only the prefixes that reach it are kept from the filter
@pytest.mark.parametrize("value", [np.nan, -np.inf, 1e-21, 3e19])
def test_rows_without_a_norm(P, value):
    data = synthdata.small(20000, 2048, 256, 64, 45)
    db = data["db"].copy()
    if value == 1e-21:
        db[777] = 0
    db[777, 255] = value
    g = P.index_create(torch.from_numpy(db).cuda(), torch.from_numpy(data["means"][:16, :16].copy()).cuda(),
                       torch.arange(20000, dtype=torch.int32, device="cuda") % 16)
    q = torch.from_numpy(data["queries"]).cuda()
    for d_s in (128, 256):
        P.profile_enable(True)
        a = [t.cpu().numpy() for t in P.search_ivf(g, q, 16, d_s, 8, 20)]
        stages = P.profile_read()
        P.profile_enable(False)
        assert ("mma" in stages) == (d_s == 128)
        with P.option(P.OPT_FP32_STREAM, 0):
            b = [t.cpu().numpy() for t in P.search_ivf(g, q, 16, d_s, 8, 20)]
        np.testing.assert_array_equal(a[0], b[0])
        np.testing.assert_array_equal(a[1].view(np.int32), b[1].view(np.int32))
    g.free()


# an index small enough to keep the filter: the row's lists leave their queries, and
# with them all others, to the tiled scan
@pytest.mark.parametrize("value", [np.nan, np.inf, -3e19, 1e-21])
def test_rows_without_a_norm_in_the_filter(P, value):
    data = synthdata.small(6000, 333, 64, 24, 46)
    db, q = data["db"].copy(), data["queries"].copy()
    db[11], db[77, 3], q[5] = 0, value, 0
    db[11, 0] = value
    g = P.index_create(torch.from_numpy(db).cuda(), torch.from_numpy(data["means"][:24, :16].copy()).cuda(),
                       torch.arange(6000, dtype=torch.int32, device="cuda") % 24)
    q = torch.from_numpy(q).cuda()
    P.profile_enable(True)
    a = [t.cpu().numpy() for t in P.search_ivf(g, q, 16, 64, 24, 100)]
    stages = P.profile_read()
    P.profile_enable(False)
    assert "mma" in stages
    with P.option(P.OPT_FP32_STREAM, 0):
        b = [t.cpu().numpy() for t in P.search_ivf(g, q, 16, 64, 24, 100)]
    g.status()
    np.testing.assert_array_equal(a[0], b[0])
    np.testing.assert_array_equal(a[1].view(np.int32), b[1].view(np.int32))
    g.free()
