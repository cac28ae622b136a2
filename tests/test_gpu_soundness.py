"""Calls off the beaten path on the GPU: clusters that start late, buffers and arguments of unusual
kinds, scales at the ends of the float range."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("b", [1, 128, 129, 700, 1024, 1025, 5000])
def test_kl_statistics_while_the_chip_is_full(b):
    """The CTAs of a statistics cluster start as SMs come free of another stream's work: every launch's
    mean and maximum must still be those of its rows."""
    import paper_2211_15023_b200 as P
    rng = np.random.default_rng(b)
    zo = (rng.standard_normal((b, 6)) * 2).astype(np.float32)
    zs = (zo + 0.3 * rng.standard_normal((b, 6))).astype(np.float32)
    want = oracle.kl(zo, zs)
    do, ds = torch.from_numpy(zo).cuda(), torch.from_numpy(zs).cuda()
    side = torch.cuda.Stream()
    x = torch.randn((1 << 22,), device="cuda")
    torch.cuda.synchronize()
    got = []
    for i in range(40):
        with torch.cuda.stream(side):
            x = x * 1.0000001 + 1e-9
        got.append(P.kl(do, ds)[1])
    torch.cuda.synchronize()
    # double sums of at most 5000 rows, rounded to float once
    np.testing.assert_allclose(torch.stack(got).cpu().numpy(), np.tile([want.mean(), want.max()], (40, 1)), rtol=1e-5, atol=1e-6)
