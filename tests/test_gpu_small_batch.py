"""Small batches take their own kernels (cluster mapping, probe plan, list scan,
selection); their results equal those of the same queries in a large batch,
bit for bit, and the probes those of the tensor-core cluster mapping."""
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
    data = synthdata.small(30000, 4100, 256, 48, 17)
    db = torch.from_numpy(data["db"]).cuda()
    g = P.build_ivf(db, 32, 400, 3, 8000, 3, storage=P.STORE_F32 | P.STORE_BF16)
    P.build_opq(g, db, 64, 16, 0, 1, 1, 4000, 7)
    yield g, torch.from_numpy(data["queries"]).cuda()
    g.free()


def cut(search, q, size):
    parts = [search(q[i:i + size].contiguous()) for i in range(0, q.shape[0], size)]
    return [torch.cat(t).cpu().numpy() for t in zip(*parts)]


def same(a, b):
    for x, y in zip(a, b):
        np.testing.assert_array_equal(x.view(np.int32) if x.dtype == np.float32 else x,
                                      y.view(np.int32) if y.dtype == np.float32 else y)


# pieces on both sides of the small plan (16,384 pairs), of the 64-member units
# (155,648 members) and of the 1,024-thread selection (one query per SM)
@pytest.mark.parametrize("d_s,nprobe,k,sizes", [
    (8, 1, 1, (1, 333)), (64, 32, 10, (1, 60, 511, 513)), (96, 5, 100, (7, 152, 153)),
    (256, 16, 1000, (3, 129)), (256, 400, 20, (2, 40, 41)), (48, 33, 50, (1, 300))])
def test_fp32_pieces(P, index, d_s, nprobe, k, sizes):
    g, q = index
    q = q[:600]
    f = lambda x: P.search_ivf(g, x, 32, d_s, nprobe, k, return_probes=True)
    whole = cut(f, q, 600)
    for size in sizes:
        same(cut(f, q, size), whole)


def test_probes_equal_tensor_core_mapping(P, index):
    g, q = index  # 4,100 x 400 x 32 centroid coordinates: the tensor-core mapping
    f = lambda x: P.search_ivf(g, x, 32, 64, 20, 5, storage=P.STORE_BF16, rerank_k=20,
                               return_probes=True)
    same(cut(f, q, 4100)[2:], cut(f, q, 100)[2:])


def test_other_searches_in_pieces(P, index):
    g, q = index
    q = q[:520]
    for f in (lambda x: P.search_ivf(g, x, 16, 256, 12, 10, storage=P.STORE_BF16, rerank_k=3000 // 2),
              lambda x: P.search_ivfopq(g, x, 32, 9, 10, rerank_k=0),
              lambda x: P.search_ivfopq(g, x, 32, 60, 10, rerank_k=40)):
        whole = cut(f, q, 520)
        same(cut(f, q, 1), whole)
        same(cut(f, q, 77), whole)


@pytest.mark.parametrize("metric", [0, 1])
def test_budgets_in_pieces(P, metric):
    data = synthdata.small(9000, 260, 128, 24, 5)
    g = P.build_ivf(torch.from_numpy(data["db"]).cuda(), 16, 40, 3, 9000, 3, metric=metric)
    q = torch.from_numpy(data["queries"]).cuda()
    rng = np.random.default_rng(3)
    ds = rng.choice([8, 48, 96, 128], 260).tolist()
    npr, k = rng.integers(1, 20, 260).tolist(), rng.integers(1, 60, 260).tolist()
    k[0] = 60

    def run(i, n):
        sl = slice(i, i + n)
        return P.search_ivf_budgets(g, q[sl].contiguous(), 16, ds[sl], npr[sl], k[sl], k_max=60)

    whole = [t.cpu().numpy() for t in run(0, 260)]
    for n in (1, 13):
        same([torch.cat(t).cpu().numpy() for t in zip(*[run(i, n) for i in range(0, 260, n)])],
             whole)
    g.free()
