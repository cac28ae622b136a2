"""GPU parity at the sizes where the kernels' tiles, rings and clusters end: vector-observation
networks, the KL indicators, V-trace and the checks of the native calls -- against the CPU oracle,
at the tolerances of the other parity tests (logits and codes bit for bit)."""
import numpy as np
import pytest

import oracle
import workloads as W
from parity_util import ATOL, RTOL, compare

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _mlp(dims, seed):
    rng = np.random.default_rng(seed)
    layers = W.mlp(dims)
    calib = rng.standard_normal((64, dims[0])).astype(np.float32)
    return oracle.calibrate("f32", (dims[0], 1, 1), layers, W.parameters_for(layers, seed), calib)


@pytest.mark.parametrize("dims", [[5, 256, 256, 256, 256, 3], [33, 40, 17, 2], [256, 255, 31, 32], [1, 1],
                                  [3, 128, 64, 7]], ids=lambda d: "-".join(map(str, d)))
def test_mlp_widths_and_depths(dims):
    """Widths that are no multiple of an instruction's columns or K step, one layer only, and networks
    whose weights pass through the two-slot ring; batches around both row tiles, taps included."""
    import paper_2211_15023_b200 as P
    pol = _mlp(dims, sum(dims))
    for b, flags in ((1, 1), (17, 5), (33, 0), (4800, 0)):
        rng = np.random.default_rng(b)
        obs = rng.standard_normal((b, dims[0])).astype(np.float32)
        u = rng.random(b, dtype=np.float32)
        ref = oracle.forward(pol, obs, u, keep=b < 100)
        g = P.Policy(pol, b, flags=flags)
        out = [t.cpu().numpy() for t in g.act(torch.from_numpy(obs).cuda(), torch.from_numpy(u).cuda())]
        g.check()
        compare(ref, *out, taps=g.read_activation if flags else None)
        g.close()


@pytest.mark.parametrize("b,a", [(127, 18), (128, 18), (129, 3), (1024, 18), (1025, 2), (2048, 9), (2049, 18), (2048, 6), (2049, 6), (1025, 7), (300, 64),
                                 (300, 65), (70001, 5)])
def test_kl_at_the_edges_of_blocks_and_clusters(b, a):
    import paper_2211_15023_b200 as P
    rng = np.random.default_rng(b + a)
    zo = (rng.standard_normal((b, a)) * 3).astype(np.float32)
    zs = (zo + rng.standard_normal((b, a)) * rng.choice([1e-3, 0.5, 4.0], size=(b, 1))).astype(np.float32)
    zs[b // 2] = zo[b // 2]
    want = oracle.kl(zo, zs)
    kl, stats = (t.cpu().numpy() for t in P.kl(torch.from_numpy(zo).cuda(), torch.from_numpy(zs).cuda()))
    np.testing.assert_allclose(kl, want, rtol=RTOL, atol=ATOL)
    assert kl[b // 2] == 0.0
    np.testing.assert_allclose(stats, [want.mean(), want.max()], rtol=RTOL, atol=ATOL)


@pytest.mark.parametrize("spread", [1e-6, 1.0, 100.0, 700.0, 3000.0])
def test_kl_exponentials_over_their_range(spread):
    """Differences of logits from nothing to far below the least exponential, exact zeros, infinities and NaNs."""
    import paper_2211_15023_b200 as P
    rng = np.random.default_rng(int(spread))
    zo, zs = ((rng.random((300, 18)) * spread).astype(np.float32) for _ in range(2))
    zs[::7] = zo[::7]
    want = oracle.kl(zo, zs)
    got = P.kl(torch.from_numpy(zo).cuda(), torch.from_numpy(zs).cuda())[0].cpu().numpy()
    np.testing.assert_allclose(got, want, rtol=RTOL, atol=ATOL)
    assert (got[::7] == 0.0).all()
    zo[5, 3] = zs[6, 0] = np.nan
    zo[8, 1] = np.inf
    got = P.kl(torch.from_numpy(zo).cuda(), torch.from_numpy(zs).cuda())[0].cpu().numpy()
    assert np.isnan(got[[5, 6, 8]]).all() and np.isfinite(np.delete(got, [5, 6, 8])).all()


@pytest.mark.parametrize("n,b", [(15, 31), (16, 32), (17, 33), (33, 65), (64, 1)])
def test_vtrace_at_the_edges_of_chunks(n, b):
    import paper_2211_15023_b200 as P
    r = W.rollouts(n, b, seed=n + b)
    for disc in (None, r["discounts"]):
        want = oracle.vtrace(r["logp_smaller"], r["logp_original"], r["rewards"], r["values"], r["bootstrap"],
                             r["gamma"], 1.0, 1.0, disc)
        t = {k: torch.from_numpy(r[k]).cuda() for k in ("logp_smaller", "logp_original", "rewards", "values", "bootstrap")}
        vs, adv = P.vtrace(t["logp_smaller"], t["logp_original"], t["rewards"], t["values"], t["bootstrap"], r["gamma"],
                           discounts=None if disc is None else torch.from_numpy(disc).cuda())
        np.testing.assert_allclose(vs.cpu().numpy(), want["vs"], rtol=RTOL, atol=ATOL)
        np.testing.assert_allclose(adv.cpu().numpy(), want["adv"], rtol=RTOL, atol=ATOL)


def test_native_calls_refuse_what_the_python_checks_refused():
    """Tensors of the wrong type, device or layout raise as before, status codes become AccerlError,
    and a caller's own result buffers come back as the same object."""
    import paper_2211_15023_b200 as P
    g = P.Policy(_mlp([4, 8, 2], 3), 16)
    obs, u = torch.zeros((16, 4), device="cuda"), torch.zeros(16, device="cuda")
    out = g.act(obs, u)
    assert g.act(obs, u, out) is out
    for bad_obs, bad_u in ((obs.double(), u), (obs.cpu(), u), (obs.t(), u), (obs, u[:5]), (obs, u.double())):
        with pytest.raises((AssertionError, ValueError)):
            g.act(bad_obs, bad_u)
    with pytest.raises(P.AccerlError) as e:
        g.act(torch.zeros((17, 4), device="cuda"), torch.zeros(17, device="cuda"))
    assert e.value.status == 3
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        same = g.act(obs, u)
    side.synchronize()
    assert torch.equal(same[0], out[0]) and torch.equal(same[1], out[1])
    g.close()
    with pytest.raises(P.AccerlError):
        g.act(obs, u)


@pytest.mark.parametrize("name,batches", [("nature_cnn_b160", (1, 129, 1200)), ("student_cnn_b8192", (3, 700)),
                                          ("impala_resnet_b16384", (2, 149, 264)), ("lunarlander_mlp", (5, 4500))])
@pytest.mark.parametrize("value", [False, True], ids=["plain", "value_head"])
def test_noalloc_runs_the_plan_on_the_fixed_array(name, batches, value):
    """The policy's own plan with its activations in the library's array: batches up to what the array
    holds, two handles in turn so that each finds the other's bytes in it (the residual network's zero
    borders among them), against the device call."""
    import paper_2211_15023_b200 as P
    pol = W.drawn_int8_policy(name, seed=4)
    if value:
        pol["layers"][-1]["value"] = True
    big, tiny = P.Policy(pol, max(batches)), P.Policy(pol, 1)
    other = P.Policy(W.drawn_int8_policy("nature_cnn_b160", seed=5), 1)
    stream = torch.cuda.current_stream().cuda_stream
    for b in batches:
        for g, n in ((other, "nature_cnn_b160"), (tiny, name)):
            obs, u = torch.from_numpy(W.observations(n, b)).cuda(), torch.from_numpy(W.uniforms(n, b)).cuda()
            got = (torch.full((b, g.n_actions), 7.0, device="cuda"), torch.full((b,), -1, dtype=torch.int32, device="cuda"),
                   torch.full((b,), 7.0, device="cuda"))
            status = g.act_noalloc_raw(obs.data_ptr(), u.data_ptr(), b, *(t.data_ptr() for t in got), stream)
            assert status == (3 if g is other and b > 1636 else 0)
        want = big.act(obs, u)
        tiny.check()
        for x, y in zip(got, want):
            assert torch.equal(x, y)
    for g in (big, tiny, other):
        g.close()


@pytest.mark.parametrize("b,pinned", [(1, True), (200, True), (200, False), (1101, True), (1700, False)])
def test_act_host_direct_results_and_chunks(b, pinned):
    """Results written by the kernels into pinned buffers, copied into pageable ones, and batches on both
    sides of the size from which frames go in chunks; a buffer that is not 4-byte aligned for the device
    to write goes through the staging copy.  Against the device call."""
    import paper_2211_15023_b200 as P
    name = "student_cnn_b8192"
    g = P.Policy(W.drawn_int8_policy(name, seed=8), b)
    obs, u = torch.from_numpy(W.observations(name, b, seed=b)), torch.from_numpy(W.uniforms(name, b, seed=b))
    want = [t.cpu() for t in g.act(obs.cuda(), u.cuda())]
    pin = (lambda t: t.pin_memory()) if pinned else (lambda t: t)
    for _ in range(2):
        out = (pin(torch.zeros((b, g.n_actions))), pin(torch.zeros(b, dtype=torch.int32)), pin(torch.zeros(b)))
        g.act_host(pin(obs), pin(u), out)
        for x, y in zip(out, want):
            assert torch.equal(x, y)
    raw = torch.zeros(4 * b + 1, dtype=torch.uint8).pin_memory()[1:]  # log-probs at an odd address
    g.act_host(pin(obs), pin(u), (out[0], out[1], raw))
    assert raw.numpy().tobytes() == want[2].numpy().tobytes()
    g.check()
    g.close()


@pytest.mark.parametrize("small,orig,b", [("student_cnn_b8192", "nature_cnn_b160", 1), ("student_cnn_b8192", "nature_cnn_b160", 2300),
                                          ("student_cnn_b8192", "impala_resnet_b16384", 1100), ("impala_resnet_b16384", "nature_cnn_b160", 460)])
@pytest.mark.parametrize("alpha", [0.0, 0.07, 0.8, 1.0])
def test_mixing_routes_every_state_through_its_network(small, orig, b, alpha):
    """States listed per network on the device, including empty lists, lists longer and shorter than
    the host expects, and handles whose own plan runs other kernels; every state must get what its
    network alone gives, twice in a row with different selections."""
    import paper_2211_15023_b200 as P
    gs, go = P.Policy(W.drawn_int8_policy(small, seed=1), b), P.Policy(W.drawn_int8_policy(orig, seed=2), b)
    obs, u = torch.from_numpy(W.observations(small, b)).cuda(), torch.from_numpy(W.uniforms(small, b)).cuda()
    a, o = gs.act_ex(obs, u), go.act_ex(obs, u)
    for call in range(2):
        rng = np.random.default_rng(call)
        sel = rng.random(b, dtype=np.float32) if call == 0 else np.full(b, 0.06, np.float32)
        out = P.act_mixed(gs, go, obs, u, torch.from_numpy(sel).cuda(), alpha)
        gs.check()
        go.check()
        pick = torch.from_numpy(sel < np.float32(alpha)).cuda()
        assert torch.equal(out["use_smaller"].bool(), pick)
        for k in ("logits", "actions", "logp", "entropy"):
            m = pick[:, None] if k == "logits" else pick
            assert torch.equal(out[k], torch.where(m, a[k], o[k])), k
    gs.close()
    go.close()


@pytest.mark.parametrize("name,b", [("nature_cnn_b160", 149), ("nature_cnn_b160", 297), ("nature_cnn_b160", 600),
                                    ("student_cnn_b8192", 148), ("student_cnn_b8192", 745)])
def test_atari_kernel_with_one_two_and_three_images_per_context(name, b):
    """Batches around one, two and three images per SM and beyond, where CTAs have one to three contexts
    and contexts one to three images, some CTAs one image less than others."""
    import paper_2211_15023_b200 as P
    pol = W.drawn_int8_policy(name, seed=11)
    obs, u = W.observations(name, b, seed=b), W.uniforms(name, b, seed=b)
    ref = oracle.forward(pol, obs, u, keep=False)
    g = P.Policy(pol, b)
    assert "atari_kernel" in g.info()["plan"]
    for _ in range(2):
        out = [t.cpu().numpy() for t in g.act(torch.from_numpy(obs).cuda(), torch.from_numpy(u).cuda())]
        g.check()
        compare(ref, *out)
    g.close()


@pytest.mark.parametrize("hidden,actions,value,b", [(16, 1, False, 1), (80, 8, False, 17), (208, 7, True, 449), (48, 9, False, 31),
                                                    (240, 16, False, 100), (64, 24, True, 15), (128, 31, True, 65), (144, 32, False, 16)])
def test_last_layer_and_sampler_widths(hidden, actions, value, b):
    """The launch of the last layer and the sampler on widths at the edges of its instructions' K and column
    tiles, states that are no multiple of the sixteen of a warp, with and without a value column."""
    name = "student_cnn_b8192"
    layers = W.nature_cnn(16, 32, 32, hidden, actions=actions)
    if value:
        layers = W.with_value_head(layers)
    pol = oracle.calibrate("u8", (4, 84, 84), layers, W.parameters_for(layers, hidden), W.calibration_batch(name, 16))
    obs, u = W.observations(name, b, seed=b), W.uniforms(name, b, seed=b)
    ref = oracle.forward(pol, obs, u, keep=False)
    import paper_2211_15023_b200 as P
    g = P.Policy(pol, b)
    assert "fc_sample_kernel covers layer 4+sample" in g.info()["plan"]
    out = {k: v.cpu().numpy() for k, v in g.act_ex(torch.from_numpy(obs).cuda(), torch.from_numpy(u).cuda()).items()}
    g.check()
    compare(ref, out["logits"], out["actions"], out["logp"], value=out.get("value"), entropy=out["entropy"])
    g.close()


@pytest.mark.parametrize("hidden,actions,value,b", [(256, 18, False, 641), (256, 3, True, 2049), (256, 32, False, 4737), (256, 8, True, 9473),
                                                    (512, 18, True, 449), (512, 31, False, 2176), (512, 6, False, 4737), (512, 5, False, 9500)])
def test_hidden_layer_last_layer_and_sampler_in_tiles(hidden, actions, value, b):
    """The launch that ends larger steps at every number of CTAs per tile of states, ragged last tiles, and one
    state more than it takes (9500 of 512 outputs); device calls, the fixed workspace and routed states."""
    import paper_2211_15023_b200 as P
    name, n = "student_cnn_b8192", 300
    layers = W.nature_cnn(16, 32, 32, hidden, actions=actions)
    if value:
        layers = W.with_value_head(layers)
    pol = oracle.calibrate("u8", (4, 84, 84), layers, W.parameters_for(layers, hidden), W.calibration_batch(name, 16))
    obs, u = W.observations(name, n, seed=b), W.uniforms(name, n, seed=b)
    ref = oracle.forward(pol, obs, u, keep=False)
    at = np.random.default_rng(b).integers(0, n, b)  # the states of the batch, drawn from those
    ref = {k: v[at] if isinstance(v, np.ndarray) and len(v) == n else v for k, v in ref.items()}
    g = P.Policy(pol, b)
    assert ("fc_tile_fc_sample_kernel" in g.info()["plan"]) == (b != 9500)
    obs, u = torch.from_numpy(obs).cuda()[torch.from_numpy(at).cuda()], torch.from_numpy(u[at]).cuda()
    res = g.act_ex(obs, u)
    g.check()
    out = {k: v.cpu().numpy() for k, v in res.items()}
    compare(ref, out["logits"], out["actions"], out["logp"], value=out.get("value"), entropy=out["entropy"])
    if b < 1000:  # (the fixed workspace ends at some 1600 of them)
        got = [torch.empty_like(res[k]) for k in ("logits", "actions", "logp")]
        stream = torch.cuda.current_stream().cuda_stream
        assert g.act_noalloc_raw(obs.data_ptr(), u.data_ptr(), b, *(t.data_ptr() for t in got), stream) == 0
        for k, t in zip(("logits", "actions", "logp"), got):
            assert torch.equal(t, res[k]), k
    if b <= 2176:
        other = P.Policy(pol, b)
        mixed = P.act_mixed(g, other, obs, u, torch.rand(b, device="cuda"), 0.4)
        g.check()
        other.check()
        for k in ("logits", "actions", "logp"):
            assert torch.equal(mixed[k], res[k]), k
        other.close()
    g.close()


def _requantisers(g, kernel):
    """For each launch of ``kernel`` in the plan: "A" if layers run the single-fma requantiser, "D" if layers run the
    three-step division, "AD" for some of each."""
    return [("A" if "single-fma requantiser verified" in l else "") + ("D" if "3-step divide verified" in l else "")
            for l in g.info()["plan"].splitlines() if kernel in l]


# drawn residual networks: every layer with single-fma constants (the kernels without the division's code), layers of
# both sorts in two launches and none in the first, the search skipped
RESIDUAL_FORMS = {"single_fma": (1, "", ["A", "A", "A"]), "both": (2, "", ["D", "AD", "AD"]),
                  "division": (21, "FLAG_TEST_NO_AFFINE", ["D", "D", "D"])}


@pytest.mark.parametrize("b", [1, 148, 149, 445, 900])
@pytest.mark.parametrize("form", list(RESIDUAL_FORMS))
def test_residual_network_kernels_by_images_per_sm(b, form):
    """One image per SM, two or three at once, several in turn; single-fma code, code with both requantisers, division in
    every layer: the logits of the dp4a kernels, bit for bit."""
    import paper_2211_15023_b200 as P
    seed, flag, want = RESIDUAL_FORMS[form]
    pol = W.drawn_int8_policy("impala_resnet_b16384", seed=seed)
    obs = torch.from_numpy(W.observations("impala_resnet_b16384", b, seed=b)).cuda()
    u = torch.from_numpy(W.uniforms("impala_resnet_b16384", b, seed=b)).cuda()
    got = []
    for flags in (getattr(P, flag) if flag else 0, P.FLAG_FORCE_GENERIC):
        g = P.Policy(pol, b, flags=flags)
        assert _requantisers(g, "res_") == ([] if flags == P.FLAG_FORCE_GENERIC else want), g.info()["plan"]
        got.append([t.clone() for t in g.act(obs, u)])
        g.check()
        g.close()
    for x, y in zip(*got):
        assert torch.equal(x, y)


@pytest.mark.parametrize("b", [5, 149, 460])
@pytest.mark.parametrize("form", list(RESIDUAL_FORMS))
def test_residual_network_activations_by_images_per_sm(b, form):
    """The same kernels with the stores of their taps, at one image per SM, at two, and where contexts take several in
    turn: every tensor that the plan stores is the dp4a kernels', bit for bit."""
    import paper_2211_15023_b200 as P
    seed, flag, want = RESIDUAL_FORMS[form]
    name = "impala_resnet_b16384"
    pol = W.drawn_int8_policy(name, seed=seed)
    obs = torch.from_numpy(W.observations(name, b, seed=b)).cuda()
    u = torch.from_numpy(W.uniforms(name, b, seed=b)).cuda()
    g = P.Policy(pol, b, flags=P.FLAG_KEEP_ACTIVATIONS | P.FLAG_TAP_FUSED | (getattr(P, flag) if flag else 0))
    ref = P.Policy(pol, b, flags=P.FLAG_KEEP_ACTIVATIONS | P.FLAG_FORCE_GENERIC)
    assert _requantisers(g, "res_") == want, g.info()["plan"]
    for x, y in zip(g.act(obs, u), ref.act(obs, u)):
        assert torch.equal(x, y)
    g.check()
    missing = []
    for i in range(-1, len(pol["layers"]) - 1):
        try:
            got = g.read_activation(i, b)
        except P.AccerlError as e:
            assert e.status == 2
            missing.append(i)
            continue
        assert np.array_equal(got, ref.read_activation(i, b)), "layer %d" % i
    assert missing == [0, 6, 17]  # pooled before they are stored, or kept ReLU'd only
    g.close()
    ref.close()


@pytest.mark.parametrize("seed,flag,want", [(1, "", ["A", "A"]), (22, "", ["D", "A"]), (22, "FLAG_TEST_NO_AFFINE", ["D", "D"])],
                         ids=["single_fma", "division_and_single_fma", "division"])
def test_conv_rows_by_batch(seed, flag, want):
    """Fewer grid rows than a tile holds, whole tiles and remainders, fewer and more steps than SMs: the logits of the
    dp4a kernels, bit for bit."""
    import paper_2211_15023_b200 as P
    name, top = "nature_cnn_b8192", 2561  # above the single-launch conv stack
    pol = W.drawn_int8_policy(name, seed=seed)
    g, ref = P.Policy(pol, top, flags=getattr(P, flag) if flag else 0), P.Policy(pol, top, flags=P.FLAG_FORCE_GENERIC)
    assert _requantisers(g, "conv_rows_kernel") == want, g.info()["plan"]
    for b in (1, 11, 12, 13, 14, 15, 168, 200, 1000, top):
        obs = torch.from_numpy(W.observations(name, b, seed=b)).cuda()
        u = torch.from_numpy(W.uniforms(name, b, seed=b)).cuda()
        for x, y in zip(g.act(obs, u), ref.act(obs, u)):
            assert torch.equal(x, y)
    g.check()
    g.close()
    ref.close()


@pytest.mark.parametrize("a", [1, 2, 3, 4, 7, 12, 17, 18, 20, 24])
def test_kl_rows_by_width_and_alignment(a):
    """Rows copied 16 bytes at a time and read 1, 2 or 4 elements at a time, the last block's remainder among them,
    against the same rows at an address that is no multiple of 16 bytes: the same bits.  (Up to 2048 rows of at most six
    actions go to the single launch, which always copies element by element.)"""
    import paper_2211_15023_b200 as P
    b = max(256 * a, 2048) + 131
    rng = np.random.default_rng(a)
    z = torch.from_numpy(rng.standard_normal((2, b * a), np.float32) * 3).cuda()
    odd = torch.empty((2, b * a + 8), device="cuda")
    shifted = [odd[i].view(-1)[1:1 + b * a] for i in range(2)]
    for d, s in zip(shifted, z):
        d.copy_(s)
    assert z[0].data_ptr() % 16 == 0 and shifted[0].data_ptr() % 16 == 4
    zo, zs = z[0].view(b, a), z[1].clone().view(b, a)
    want = P.kl(zo, zs)
    for x, y in zip(want, P.kl(shifted[0].view(b, a), shifted[1].view(b, a))):
        assert torch.equal(x, y)
    po, ps = torch.log_softmax(zo.double(), -1), torch.log_softmax(zs.double(), -1)
    np.testing.assert_allclose(want[0].cpu().numpy(), (po.exp() * (po - ps)).sum(-1).cpu().numpy(), rtol=RTOL, atol=ATOL)


@pytest.mark.parametrize("rows", [1, 37])
@pytest.mark.parametrize("c1,c2,hidden", [(5, 18, 33), (16, 70, 40), (20, 48, 300)])
def test_calibration_of_odd_shapes(rows, c1, c2, hidden):
    """Channels that fill no word, padding, strides, remainders of positions and rows: scales and codes are the
    oracle's bits."""
    import paper_2211_15023_b200 as P
    rng = np.random.default_rng(rows * 100 + c1)
    shape = (3, 17, 13)
    layers = [W._conv(3, 17, 13, c1, 5, 2, 2), W._conv(c1, 9, 7, c2, 3, 1, 1), W._conv(c2, 9, 7, 8, 7, 3, 0),
              W._fc(8, hidden), W._fc(hidden, 5, relu_out=False, logits=True)]
    params = W.parameters_for(layers, 17)
    calib = rng.integers(0, 256, (rows,) + shape, dtype=np.uint8)
    want = oracle.calibrate("u8", shape, layers, params, calib)
    g = P.Policy.from_fp32("u8", shape, layers, params, calib, 3)
    for i, l in enumerate(want["layers"]):
        got = g.export(i)
        assert got["s_in"] == np.float32(l["s_in"]) and got["s_out"] == np.float32(l["s_out"]), i
        assert np.array_equal(got["w"], l["w"]) and np.array_equal(got["s_w"], l["s_w"])
    g.close()
