"""Kernels at the ends of their ranges: the one-kernel probe plan around 8,192
(query, list) pairs and 4,096 lists, and the k-means assignment between 1,025 and
4,097 centroids.  Results equal the general kernels', bit for bit."""
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


def same(a, b):
    for x, y in zip(a, b):
        x, y = x.cpu().numpy(), y.cpu().numpy()
        np.testing.assert_array_equal(x.view(np.int32) if x.dtype == np.float32 else x,
                                      y.view(np.int32) if y.dtype == np.float32 else y)


# 8,160, 8,192 and 8,224 pairs at 32 probes, 8,000 and 8,400 at 400, 8,191 to 8,193 at 1
@pytest.mark.parametrize("nlist,nprobe,sizes", [
    (400, 32, (255, 256, 257)), (400, 400, (20, 21)), (4096, 1, (8191, 8192, 8193)),
    (4097, 1, (500,)), (4095, 16, (512, 513))])
@pytest.mark.parametrize("tier", ["f32", "bf16"])
def test_probe_plan(P, nlist, nprobe, sizes, tier):
    if tier == "bf16" and nprobe > 128:
        pytest.skip("the low-precision tiers take 128 probes")
    data = synthdata.small(20000, max(sizes), 64, 48, 19)
    rng = np.random.default_rng(nlist)
    cent = torch.from_numpy(rng.standard_normal((nlist, 16)).astype(np.float32)).cuda()
    assign = torch.from_numpy(rng.integers(0, nlist, 20000).astype(np.int32)).cuda()
    g = P.index_create(torch.from_numpy(data["db"]).cuda(), cent, assign,
                       storage=P.STORE_F32 | P.STORE_BF16)
    q = torch.from_numpy(data["queries"]).cuda()
    kw = {"storage": P.STORE_BF16, "rerank_k": 40} if tier == "bf16" else {}

    def search(x):
        return P.search_ivf(g, x, 16, 64, nprobe, 10, return_probes=True, **kw)

    for n in sizes:  # against the same rows a hundred at a time
        parts = [search(q[i:min(i + 100, n)].contiguous()) for i in range(0, n, 100)]
        same(search(q[:n].contiguous()), [torch.cat(t) for t in zip(*parts)])
    g.free()


@pytest.mark.parametrize("nc", [1025, 2048, 2049, 4095, 4096, 4097])
@pytest.mark.parametrize("dim", [16, 64])
def test_assignment(P, nc, dim):
    data = synthdata.small(9001, 8, 64, 300, nc)
    x = torch.from_numpy(data["db"]).cuda()
    cent = torch.nn.functional.normalize(x[:nc, :dim], dim=1).contiguous()
    cent[nc - 1] = cent[3]  # an equal one: the lower index wins
    a = P.kmeans_assign(x, cent, dim)
    with P.option(P.OPT_COARSE_TC, 0):
        b = P.kmeans_assign(x, cent, dim)
    same(a, b)
    assert not bool((a[0] == nc - 1).any())
