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


@pytest.mark.parametrize("n,b", [(1, 70001), (4, 1), (5, 33), (9, 16385), (16, 30001), (17, 16384), (40, 20000), (128, 4097)])
def test_vtrace_is_the_same_for_many_rollouts_as_for_few(n, b):
    """Sizes on both sides of the choice between a thread per rollout and a warp per step: against the
    oracle, and, bit for bit, against the same rollouts in slices that are stepped the other way."""
    import paper_2211_15023_b200 as P
    import workloads as W
    r = W.rollouts(n, b, seed=n + b)
    for disc in (None, r["discounts"]):
        want = oracle.vtrace(r["logp_smaller"], r["logp_original"], r["rewards"], r["values"], r["bootstrap"],
                             r["gamma"], 1.0, 1.0, disc)
        names = ("logp_smaller", "logp_original", "rewards", "values")
        t = [torch.from_numpy(r[k]).cuda() for k in names]
        boot, d = torch.from_numpy(r["bootstrap"]).cuda(), None if disc is None else torch.from_numpy(disc).cuda()
        vs, adv = P.vtrace(*t, boot, r["gamma"], discounts=d)
        np.testing.assert_allclose(vs.cpu().numpy(), want["vs"], rtol=1e-5, atol=1e-6)
        np.testing.assert_allclose(adv.cpu().numpy(), want["adv"], rtol=1e-5, atol=1e-6)
        for lo in range(0, b, max(256, b // 3)):
            part = slice(lo, min(lo + 256, b))
            some = P.vtrace(*(x[:, part].contiguous() for x in t), boot[part].contiguous(), r["gamma"],
                            discounts=None if d is None else d[:, part].contiguous())
            assert torch.equal(some[0], vs[:, part]) and torch.equal(some[1], adv[:, part])


def test_vtrace_of_short_rollouts_is_bound_by_memory():
    """A million rollouts of one step are 28 MB: 4 us at the copy rate of HBM.  The bound leaves room for a
    factor of ten; a block of a warp per time step, of which one step exists, takes 140 us."""
    import paper_2211_15023_b200 as P
    x = [torch.randn((1, 1 << 20), device="cuda") for _ in range(4)]
    boot = torch.randn(1 << 20, device="cuda")
    out = (torch.empty_like(x[0]), torch.empty_like(x[0]))
    best = 1e9
    for _ in range(5):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        P.vtrace(*x, boot, 0.99, out=out)
        a.record()
        for _ in range(20):
            P.vtrace(*x, boot, 0.99, out=out)
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b) * 50.0)
    assert best < 50.0, "%.1f us" % best
