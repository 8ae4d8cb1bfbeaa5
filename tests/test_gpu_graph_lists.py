"""Graph search at every register list size, degree and prefix against a plain
best-first search on the CPU over the library's own graph.  The distances
decide the order of the expansions, so the graph is made of points whose
coordinates are small integers (raw L2): every distance is exact in FP32 and the
two must agree exactly, ties by id included."""
import heapq

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def best_first(x, q, nbr, entry, L):
    def key(i):
        return (float(((q - x[i]) ** 2).sum()), int(i))
    lst, done = [key(entry)], set()
    while True:
        cur = next((e for e in lst if e not in done), None)
        if cur is None:
            return lst
        done.add(cur)
        new = [key(u) for u in nbr[cur[1]] if u >= 0]
        lst = heapq.nsmallest(L, lst + [e for e in new if e not in set(lst)])


# list sizes at and beside the register blocks (32, 64, 128, 256, 512), degrees
# of one and two halves, rerank rows of 512, 1,024 and 2,048 coordinates
@pytest.mark.parametrize("L,R,d_g,d_s,rerank,k", [
    (1, 8, 8, 8, 1, 1), (31, 32, 16, 64, 31, 10), (32, 33, 8, 512, 20, 20), (33, 64, 16, 768, 33, 5),
    (64, 32, 64, 1024, 64, 64), (65, 16, 32, 64, 65, 3), (128, 64, 16, 2048, 128, 100),
    (200, 32, 8, 64, 200, 200), (300, 24, 16, 64, 270, 270), (512, 64, 8, 64, 400, 50)])
def test_lists_equal_best_first(L, R, d_g, d_s, rerank, k):
    import paper_2305_19435_gb300 as P
    P.build()
    N, B, d = 1500, 9, max(d_s, d_g)
    rng = np.random.default_rng(L * 7 + R)
    db = rng.integers(-3, 4, (N, d)).astype(np.float32)
    q = rng.integers(-3, 4, (B, d)).astype(np.float32)
    nbr = np.full((N, R), -1, np.int32)
    for i in range(N):
        n = rng.integers(1, R + 1)
        nbr[i, :n] = rng.choice(N, n, replace=False)
    g = P.graph_create(torch.from_numpy(db).cuda(), d_g, torch.from_numpy(nbr).cuda(), 17,
                       metric=P.METRIC_L2)
    ids, dist, short = P.graph_search(g, torch.from_numpy(q).cuda(), L, d_s, k, rerank,
                                      return_shortlist=True)
    ids, dist, short = ids.cpu().numpy(), dist.cpu().numpy(), short.cpu().numpy()
    for b in range(B):
        lst = best_first(db[:, :d_g], q[b, :d_g], nbr, 17, L)[:rerank]
        want = [i for _, i in lst] + [-1] * (rerank - len(lst))
        np.testing.assert_array_equal(short[b], want)
        full = sorted((float(((q[b, :d_s] - db[i, :d_s]) ** 2).sum()), i) for _, i in lst)[:k]
        np.testing.assert_array_equal(ids[b], [i for _, i in full] + [-1] * (k - len(full)))
        np.testing.assert_array_equal(dist[b], np.float32([v for v, _ in full] +
                                                          [np.inf] * (k - len(full))))
    g.free()
