"""Which route an IVF-OPQ batch takes with few queries per list and short rows: the
tensor-core filter only where both sides' estimates put it ahead.  The scores and
ids are the running top-k scan's, bit for bit, on both."""
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
    data = synthdata.small(100_000, 800, 128, 256, 47)
    db = torch.from_numpy(data["db"]).cuda()
    g = P.build_ivf(db, 16, 400, 3, 20000, 3)
    yield g, db, torch.from_numpy(data["queries"]).cuda()
    g.free()


# 19, 33 and 33 queries per list
@pytest.mark.parametrize("d_s,M,nprobe,k,B,filtered", [
    (64, 32, 51, 1, 150, False), (128, 64, 17, 6, 781, True), (64, 8, 17, 6, 781, False)])
def test_route(P, index, d_s, M, nprobe, k, B, filtered):
    g, db, q = index
    q = q[:B]
    R = torch.linalg.qr(torch.randn(d_s, d_s, device="cuda"))[0].contiguous()
    z = torch.nn.functional.normalize(db[:256, :d_s], dim=1) @ R
    C = z.view(256, M, d_s // M).transpose(0, 1).contiguous()
    P.set_opq(g, d_s, M, R, C, P.opq_encode(db, d_s, M, R, C))
    P.profile_enable(True)
    a = [t.cpu().numpy() for t in P.search_ivfopq(g, q, 16, nprobe, k)]
    stages = P.profile_read()
    P.profile_enable(False)
    assert ("mma" in stages) == filtered
    with P.option(P.OPT_ADC_SELECT, 0):
        b = [t.cpu().numpy() for t in P.search_ivfopq(g, q, 16, nprobe, k)]
    np.testing.assert_array_equal(a[0], b[0])
    np.testing.assert_array_equal(a[1].view(np.int32), b[1].view(np.int32))
