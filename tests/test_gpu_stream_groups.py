"""The streaming FP32 scan's groups of queries: every filling of a tile of 16
queries and of a group of 8, lists that end inside a unit of 128 members, partial
blocks (d_s 8) and rows for which fewer queries are staged (d_s 2048) give the
tiled scan's ids and distances, bit for bit."""
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


@pytest.fixture(scope="module", params=[0, 1])
def index(P, request):
    data = synthdata.small(6000, 700, 2048, 40, 23)
    g = P.build_ivf(torch.from_numpy(data["db"]).cuda(), 16, 60, 3, 6000, 3, metric=request.param)
    yield g, torch.from_numpy(data["queries"]).cuda()
    g.free()


def same(a, b):
    for x, y in zip(a, b):
        assert torch.equal(x.view(torch.int32) if x.dtype == torch.float32 else x,
                           y.view(torch.int32) if y.dtype == torch.float32 else y)


# 560 x 3 to 700 x 9 pairs over 60 lists, about 100 members each: past the small
# batches' kernel (155,648 members), on both sides of 16 queries per list; k 300
# keeps to these scans
@pytest.mark.parametrize("d_s,B,nprobe", [(8, 640, 3), (48, 560, 3), (512, 700, 9), (1024, 640, 5),
                                          (2048, 560, 3)])
def test_groups_equal_tiled_scan(P, index, d_s, B, nprobe):
    g, q = index
    got = P.search_ivf(g, q[:B].contiguous(), 16, d_s, nprobe, 300)
    with P.option(P.OPT_FP32_STREAM, 0):
        want = P.search_ivf(g, q[:B].contiguous(), 16, d_s, nprobe, 300)
    same(got, want)


def test_mixed_prefixes_equal_single_prefix_calls(P, index):
    g, q = index
    rng = np.random.default_rng(9)
    grid = [8, 16, 48, 512, 2048]
    ds = rng.choice(grid, 700)
    npr, k = rng.integers(1, 9, 700), rng.integers(1, 300, 700)
    k[0] = 300
    ids, dist = P.search_ivf_budgets(g, q, 16, ds.tolist(), npr.tolist(), k.tolist())
    for i in range(0, 700, 7):
        with P.option(P.OPT_FP32_STREAM, 0):
            wi, wd = P.search_ivf(g, q[i:i + 1].contiguous(), 16, int(ds[i]), int(npr[i]), int(k[i]))
        same((ids[i, :k[i]], dist[i, :k[i]]), (wi[0], wd[0]))
