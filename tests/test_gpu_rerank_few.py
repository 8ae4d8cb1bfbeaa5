"""Short shortlists (up to 32 slots, of short rows up to 64) are re-scored and sorted several queries to a
CTA; results equal, bit for bit, those of a longer shortlist's kernels where both
hold every candidate."""
import numpy as np
import pytest

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


# lists of 3 to 7 members: at most 7 candidates per probe; one query, a query, four
# and sixteen per CTA, the last CTA part-filled (enough rows that the shortlists are
# re-scored query by query)
@pytest.mark.parametrize("d_s", [8, 64, 96, 1024, 2048])
def test_equals_longer_shortlists(P, d_s):
    N, d = (140_000 if d_s < 512 else 50_000), max(d_s, 64)
    gen = torch.Generator(device="cuda").manual_seed(d_s)
    db = torch.randn(N, d, device="cuda", generator=gen)
    size = 3 + torch.arange(N // 5 + 2, device="cuda") % 5
    assign = torch.repeat_interleave(torch.arange(len(size), device="cuda"), size)[:N].int()
    assign = assign[torch.randperm(N, device="cuda", generator=gen)].contiguous()
    nlist = int(assign.max()) + 1
    assert nlist <= 32768 and int(torch.bincount(assign.long()).max()) <= 7
    cent = torch.nn.functional.normalize(torch.randn(nlist, 16, device="cuda", generator=gen))
    g = P.index_create(db, cent, assign, storage=P.STORE_F32 | P.STORE_BF16 | P.STORE_FP8)
    queries = torch.randn(35_003, d, device="cuda", generator=gen)
    batches = [(1, 4, 31, 65), (333, 4, 31, 65), (9001, 4, 30, 65), (35_003, 1, 8, 66)]
    if d_s <= 128:  # up to 64 slots, of 56 candidates
        batches += [(1, 8, 64, 65), (2001, 8, 57, 90), (4100, 8, 62, 65)]
    for B, npb, few, many in batches:
        q = queries[:B].contiguous()
        for tier in (P.STORE_BF16, P.STORE_FP8):
            for k in (1, few - 1):
                f = lambda rr: P.search_ivf(g, q, 16, d_s, npb, k, storage=tier, rerank_k=rr)
                same(f(few), f(many))
    if d_s <= 96:
        M = d_s // 8
        R = torch.eye(d_s, device="cuda")
        z = torch.nn.functional.normalize(db[:256, :d_s], dim=1)
        C = z.view(256, M, 8).transpose(0, 1).contiguous()
        P.set_opq(g, d_s, M, R, C, P.opq_encode(db, d_s, M, R, C))
        for B, npb, few, many in batches + [(9001, 4, 32, 70)]:
            q = queries[:B].contiguous()
            for k in (1, few):
                f = lambda rr: P.search_ivfopq(g, q, 16, npb, k, rerank_k=rr)
                same(f(few), f(many))
                np1, kq = [1 + i % npb for i in range(B)], [1 + i % k for i in range(B)]
                kq[0] = k
                h = lambda rr: P.search_ivfopq_budgets(g, q, 16, np1, kq, rerank_k=rr)
                same(h(few), h(many))
    g.status()
    g.free()
