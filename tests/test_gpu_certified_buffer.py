"""The certified shortlist's buffer: lists whose sampled keys are all far, so that
the sampled threshold lets nearly every key in and the buffer of 1,024 fills
and is tightened over and over, at lengths around the pipeline's halves (1,536
and 2,560 keys for many and few queries).  The results equal the tiled scan's bit
for bit, and the queries whose certified set fits are answered by the filter."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def arc_rows(n, far, rng):
    """Unit vectors on an arc, angle (and distance to the arc's start) in random order over the
    positions, those in `far` opposite to it."""
    a = np.linspace(0.02, 1.4, n)[rng.permutation(n)]
    a[far] = np.pi - 0.3 * rng.random(len(far))
    x = np.zeros((n, 16), np.float32)
    x[:, 0], x[:, 1] = np.cos(a), np.sin(a)
    return x


def sampled(n):
    """Positions of the 256 runs of 8 keys that the threshold is taken from."""
    nvec = (n + 7) // 8
    step = (nvec << 20) // 256
    return np.concatenate([8 * ((j * step) >> 20) + np.arange(8) for j in range(256)])


@pytest.mark.parametrize("B", [1200, 1300])  # on both sides of 8 queries per SM
@pytest.mark.parametrize("n", [3071, 3072, 3073, 4608, 5120, 5121, 7680, 7681])
def test_buffer_fills_and_tightens(n, B):
    import paper_2305_19435_gb300 as P
    P.build()
    rng = np.random.default_rng(n)
    far = np.unique(np.minimum(sampled(n), n - 1))
    x = arc_rows(n, far, rng)
    phi = 0.3 * rng.random(B)
    q = np.zeros((B, 16), np.float32)
    q[:, 0], q[:, 1] = np.cos(phi), np.sin(phi)
    q[::50] = 0  # every member equally near: left over
    g = P.flat_index(torch.from_numpy(x).cuda())
    q = torch.from_numpy(q).cuda()
    for k in (2, 10, 100):
        P.profile_enable(True)
        a = [t.cpu().numpy() for t in P.search_ivf(g, q, 8, 16, 1, k)]
        prof = P.profile_read()
        P.profile_enable(False)
        g.status()
        assert "mma" in prof
        with P.option(P.OPT_FP32_STREAM, 0):
            b = [t.cpu().numpy() for t in P.search_ivf(g, q, 8, 16, 1, k)]
        np.testing.assert_array_equal(a[0], b[0])
        np.testing.assert_array_equal(a[1].view(np.int32), b[1].view(np.int32))
    g.free()
