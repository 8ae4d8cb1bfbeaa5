"""The rerank's routes agree bit for bit: shortlists re-scored member by member
(many slots per database row), query by query, split over CTAs (few queries)
and with the queries taken in list order (large batches)."""
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


def in_pieces(search, q, size):
    parts = [search(q[i:i + size]) for i in range(0, q.shape[0], size)]
    return [torch.cat(t).cpu().numpy() for t in zip(*parts)]


def check(search, q, size):
    whole, cut = [t.cpu().numpy() for t in search(q)], in_pieces(search, q, size)
    np.testing.assert_array_equal(whole[0], cut[0])
    np.testing.assert_array_equal(whole[1].view(np.int32), cut[1].view(np.int32))


# coordinate groups below, at and above a lane's eight loads; shortlists below
# 256, up to 512 and above (the final sort's three forms); an empty-slot case
# (rerank_k beyond the candidates)
@pytest.mark.parametrize("tier,d,d_s,k,rerank,size", [
    ("BF16", 64, 8, 5, 20, 31), ("FP8", 96, 96, 10, 300, 64), ("BF16", 512, 512, 100, 400, 7),
    ("FP8", 2048, 2048, 20, 80, 100), ("BF16", 768, 768, 100, 600, 1),
    ("FP8", 256, 256, 50, 2048, 40)])
def test_by_query_equals_by_member(P, tier, d, d_s, k, rerank, size):
    data = synthdata.small(1500, 700, d, 16, d_s)
    store = getattr(P, "STORE_" + tier)
    g = P.build_ivf(torch.from_numpy(data["db"]).cuda(), min(d, 16), 12, 3, 1500, 5,
                    storage=P.STORE_F32 | store)
    q = torch.from_numpy(data["queries"]).cuda()
    check(lambda x: P.search_ivf(g, x.contiguous(), min(d, 16), d_s, 4, k, storage=store,
                                 rerank_k=rerank), q, size)
    g.free()


def test_list_order(P):
    """Batches large enough to be taken in list order (BF16 and IVF-OPQ)."""
    data = synthdata.small(60000, 2200, 512, 32, 3)
    db = torch.from_numpy(data["db"]).cuda()
    g = P.build_ivf(db, 32, 40, 3, 20000, 5, storage=P.STORE_F32 | P.STORE_BF16)
    P.build_opq(g, db, 512, 32, 0, 1, 1, 4000, 7)
    q = torch.from_numpy(data["queries"]).cuda()
    check(lambda x: P.search_ivf(g, x.contiguous(), 32, 512, 4, 100, storage=P.STORE_BF16,
                                 rerank_k=400), q, 200)
    check(lambda x: P.search_ivfopq(g, x.contiguous(), 32, 4, 100, rerank_k=400), q, 200)
    g.free()
