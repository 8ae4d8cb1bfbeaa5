"""OPQ codes of few rows: the nearest-codeword kernel spreads the sub-vectors over
more CTAs (1, 2, 4 or 8 each); the codes equal those of the same rows in a large
block, bit for bit."""
import pytest

import synthdata

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# 32 sub-vectors in groups of 1, 2, 4 and 8; 6 and 12, where the last group is short
@pytest.mark.parametrize("M,sizes", [(32, (1, 257, 300, 2560, 5000, 9800)), (6, (3, 900, 9999)),
                                     (12, (256, 3500, 12800))])
def test_few_rows_equal_many(M, sizes):
    import paper_2305_19435_gb300 as P
    P.build()
    d_s = {32: 128, 6: 96, 12: 96}[M]
    x = torch.from_numpy(synthdata.small(30000, 8, d_s, 24, M)["db"]).cuda()
    R = torch.eye(d_s, device="cuda")
    z = torch.nn.functional.normalize(x[:256], dim=1)
    C = z.view(256, M, d_s // M).transpose(0, 1).contiguous()
    whole = P.opq_encode(x, d_s, M, R, C)
    for n in sizes:
        assert torch.equal(P.opq_encode(x[7:7 + n].contiguous(), d_s, M, R, C), whole[7:7 + n])
