"""The many-row GEMM and the register-held PQ assignment against the general
kernels, through opq_encode: code bytes of a block of rows large enough for
both equal those of the same rows encoded a few at a time (the same sums in
the same order, so no tolerance applies)."""
import pytest

import synthdata

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# GEMM tiles of 64 and 128 columns with remainders (d_s 48, 96, 192), every
# register-held sub-vector size, one that is not (3, 6) and odd row counts
@pytest.mark.parametrize("d_s,M", [(8, 2), (48, 4), (48, 8), (64, 2), (96, 4), (96, 16), (96, 32),
                                   (192, 12), (192, 16), (384, 32), (128, 32)])
@pytest.mark.parametrize("metric", [0, 1])
def test_encode_blocks_equal_pieces(d_s, M, metric):
    import paper_2305_19435_gb300 as P
    P.build()
    n = 152 * 128 + 77
    data = synthdata.small(n, 8, d_s, 24, d_s + M)
    x = torch.from_numpy(data["db"]).cuda()
    gen = torch.Generator(device="cuda").manual_seed(5)
    R = torch.linalg.qr(torch.randn(d_s, d_s, device="cuda", generator=gen))[0].contiguous()
    z = x[:256] @ R
    if metric:
        z = torch.nn.functional.normalize(x[:256], dim=1) @ R
    C = z.view(256, M, d_s // M).transpose(0, 1).contiguous()
    C[:, 200] = C[:, 17]  # equal codewords: the lower one wins
    whole = P.opq_encode(x, d_s, M, R, C, metric=metric)
    pieces = torch.cat([P.opq_encode(x[i:i + 999].contiguous(), d_s, M, R, C, metric=metric)
                        for i in range(0, n, 999)])
    assert torch.equal(whole, pieces)
    assert not (whole == 200).any()
