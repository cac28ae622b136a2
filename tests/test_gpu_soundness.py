"""Calls off the beaten path on the GPU: clusters that start late, buffers and arguments of unusual
kinds, scales at the ends of the float range."""
import numpy as np
import pytest

import oracle
from parity_util import compare

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


@pytest.mark.parametrize("a", [1, 5, 6, 7, 9, 12, 13, 18, 33, 63, 64, 65])
def test_kl_of_few_rows_and_of_many(a):
    """Row counts on both sides of every choice between one launch, a thread per row and a warp per row:
    against the oracle over spreads from nothing to far below the least exponential, and each row the same
    to the last float bit but one whichever kernel takes it (both compute in double)."""
    import paper_2211_15023_b200 as P
    rng = np.random.default_rng(a)
    b = max(256 * min(a, 64) + 130, 8193)
    zo = (rng.random((b, a)) * rng.choice([1e-6, 1.0, 100.0, 3000.0], size=(b, 1))).astype(np.float32)
    zs = (zo + rng.standard_normal((b, a)) * rng.choice([1e-3, 0.5, 50.0], size=(b, 1))).astype(np.float32)
    zs[::7] = zo[::7]
    if a > 1:  # masked actions
        zo[1::11, 0] = zs[1::11, 0] = -np.inf
        zo[2::11, 0] = zs[2::11, 0] = np.finfo(np.float32).min
    want = oracle.kl(zo, zs)
    do, ds = torch.from_numpy(zo).cuda(), torch.from_numpy(zs).cuda()
    whole = None
    for n in (b, 8193, 8192, 256 * min(a, 64), 256 * min(a, 64) - 1, 2049, 2048, 1025, 1024, 300, 1):
        n = min(n, b)
        kl, stats = (t.cpu().numpy() for t in P.kl(do[:n].contiguous(), ds[:n].contiguous()))
        np.testing.assert_allclose(kl, want[:n], rtol=1e-5, atol=1e-6)
        assert (kl[::7] == 0.0).all()
        np.testing.assert_allclose(stats, [want[:n].mean(), want[:n].max()], rtol=1e-5, atol=1e-6)
        whole = kl if whole is None else whole
        np.testing.assert_array_max_ulp(kl[kl > 1e-3], whole[:n][kl > 1e-3], maxulp=1)


def test_kl_of_few_wide_rows_does_not_wait_for_one_thread():
    """160 rows of 64 actions: a thread that walks a row of 128 exponentials takes 13 us, a warp and a second
    launch for the statistics 5.  The bound lies between them."""
    import paper_2211_15023_b200 as P
    zo = torch.randn((160, 64), device="cuda")
    zs = zo + 0.1
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        P.kl(zo, zs)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for _ in range(20):
            P.kl(zo, zs)
    best = 1e9
    for _ in range(6):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record()
        graph.replay()
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b) * 50.0)
    assert best < 10.0, "%.1f us" % best


def test_act_ex_and_act_mixed_refuse_what_their_kernels_would_misread():
    """Uniforms or selectors that are too few, of another type, on another device or strided raise on the
    host, as in act; more of them than states, which the kernels never look at, go through as before."""
    import paper_2211_15023_b200 as P
    import workloads as W
    pol, b = W.drawn_int8_policy("student_cnn_b8192"), 6
    g, o = P.Policy(pol, b), P.Policy(pol, b)
    obs = torch.from_numpy(W.observations("student_cnn_b8192", b)).cuda()
    u, long = torch.rand(b, device="cuda"), torch.rand(2 * b, device="cuda")
    bad_u = (u[:b - 1], u.double(), u.cpu(), long[::2])
    bad_obs = (obs.float(), obs.cpu(), obs.transpose(2, 3))
    for v in bad_u:
        with pytest.raises(AssertionError):
            g.act_ex(obs, v)
        with pytest.raises(AssertionError):
            P.act_mixed(g, o, obs, v, u, 0.5)
        with pytest.raises(AssertionError):
            P.act_mixed(g, o, obs, u, v, 0.5)
    for v in bad_obs:
        with pytest.raises(AssertionError):
            g.act_ex(v, u)
        with pytest.raises(AssertionError):
            P.act_mixed(g, o, v, u, u, 0.5)
    want, got = g.act_ex(obs, long[:b].contiguous()), g.act_ex(obs, long)
    for k in want:
        assert torch.equal(want[k], got[k]), k
    x, boot = torch.zeros((3, b), device="cuda"), torch.zeros(b, device="cuda")
    for call in (lambda: P.kl(x.cpu(), x.cpu()), lambda: P.kl(x, x.cpu()), lambda: P.vtrace(x, x, x, x, boot.cpu(), 0.99),
                 lambda: P.vtrace(x, x, x, x, boot, 0.99, discounts=x.double()),
                 lambda: P.vtrace(x, x, x, x, boot, 0.99, discounts=x.cpu())):
        with pytest.raises(AssertionError):
            call()
    g.check()
    g.close()
    o.close()


@pytest.mark.parametrize("b", [33, 200])
@pytest.mark.parametrize("over", ["logits", "actions", "logp"])
def test_act_host_with_the_uniforms_in_the_place_of_a_result(over, b):
    """A caller that reuses the pinned buffer of the draws for a result: the draws are all read before any
    result is written, whatever the order of the states."""
    import paper_2211_15023_b200 as P
    import workloads as W
    name = "student_cnn_b8192"
    g = P.Policy(W.drawn_int8_policy(name, seed=8), b)
    obs, u = torch.from_numpy(W.observations(name, b, seed=b)), torch.from_numpy(W.uniforms(name, b, seed=b))
    want = [t.cpu() for t in g.act(obs.cuda(), u.cuda())]
    out = dict(logits=torch.zeros((b, g.n_actions)).pin_memory(), actions=torch.zeros(b, dtype=torch.int32).pin_memory(),
               logp=torch.zeros(b).pin_memory())
    draws = out[over].view(torch.float32).reshape(-1)[:b]
    if over == "logits":
        draws = out[over].reshape(-1)[g.n_actions * b - b:]  # the last states' logits
    pinned_obs = obs.pin_memory()
    for _ in range(20):
        draws.copy_(u)
        g.act_host(pinned_obs, draws, tuple(out.values()))
        for x, y in zip(out.values(), want):
            assert torch.equal(x, y)
    g.check()
    g.close()


def _with_tiny_scale(pol, layer):
    """The policy with one layer's output on a grid so fine that the reciprocal of its scale is infinite,
    weights and the next layer's weights scaled to match."""
    tiny, ls = np.float32(1e-39), pol["layers"]
    a, b = ls[layer], ls[layer + 1]
    back = float(a["s_out"])
    a["s_w"] = (a["s_w"].astype(np.float64) * (float(tiny) / back)).astype(np.float32)  # (subnormal, a few bits each)
    a["bias"] = (a["bias"].astype(np.float64) * (float(tiny) / back)).astype(np.float32)
    a["s_out"] = b["s_in"] = tiny
    b["s_w"] = (b["s_w"].astype(np.float64) * (back / float(tiny))).astype(np.float32)
    return pol


def test_mlp_layer_whose_scale_has_no_finite_reciprocal():
    import paper_2211_15023_b200 as P
    import workloads as W
    rng = np.random.default_rng(0)
    layers = W.mlp([12, 96, 64, 5])
    params = W.parameters_for(layers, 0)
    calib = rng.standard_normal((64, 12)).astype(np.float32)
    pol = _with_tiny_scale(oracle.calibrate("f32", (12, 1, 1), layers, params, calib), 0)
    obs, u = rng.standard_normal((200, 12)).astype(np.float32), rng.random(200, dtype=np.float32)
    ref = oracle.forward(pol, obs, u)
    codes = ref["activations"][0]
    assert len(np.unique(codes)) > 20 and (codes == 127).mean() < 0.5  # (a grid that is used)
    g = P.Policy(pol, 200)
    logits, actions, logp = g.act(torch.from_numpy(obs).cuda(), torch.from_numpy(u).cuda())
    g.check()
    compare(ref, logits.cpu().numpy(), actions.cpu().numpy(), logp.cpu().numpy())
    g.close()


def test_trim_gives_back_what_is_kept_for_the_next_policy():
    """The memory of a destroyed policy stays with the library, serves the next one, and is the device's again
    after trim; a policy that is alive goes on stepping."""
    import paper_2211_15023_b200 as P
    import workloads as W
    name = "student_cnn_b8192"
    pol = W.drawn_int8_policy(name)
    obs, u = torch.from_numpy(W.observations(name, 8)).cuda(), torch.from_numpy(W.uniforms(name, 8)).cuda()
    alive = P.Policy(pol, 8)
    want = alive.act(obs, u)
    P.trim()
    free = lambda: torch.cuda.mem_get_info()[0]  # noqa: E731
    before = free()
    P.Policy(pol, 4096).close()
    kept = before - free()
    assert kept > 30 << 20
    P.Policy(pol, 4096).close()
    assert before - free() == kept
    P.trim()
    assert free() >= before
    P.trim()
    for x, y in zip(alive.act(obs, u), want):
        assert torch.equal(x, y)
    alive.check()
    alive.close()
