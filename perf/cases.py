"""Work that users of this library have it do, as cases that can be measured and compared.

An Actor process owns a compressed int8 policy and steps it once per environment step on the states
of its environments: on device buffers (``Policy.act``, ``Policy.act_ex`` where the value and the
entropy are wanted too), on host buffers (``Policy.act_host``), mixed with the original network
(``act_mixed``), or without allocating (``act_noalloc_raw``).  Beside it run the Corrector and the
Monitor on finished rollouts (``vtrace``, ``kl``), and the Compressor, which turns the Learner's
newest fp32 weights into the next int8 policy (``Policy.from_fp32``).

Networks are the repository's own: the CartPole and LunarLander perceptrons, the Atari Nature-CNN
(conv 32/64/64, fc 512), its student (16/32/32, fc 256) and the IMPALA residual network.  Batches go
from a single environment to the largest vectorised Actor; most drawn sizes are odd.
"""
import math

import numpy as np
import torch

import paper_2211_15023_b200 as P

FRAME = (4, 84, 84)


# ------------------------------------------------------------------------------- networks
def _conv(c, hw, n, k, stride, pad, relu_in=False, relu_out=True, skip=-1):
    return dict(kind="conv", in_c=c, in_h=hw, in_w=hw, out_c=n, kh=k, kw=k, stride=stride, pad=pad,
                relu_in=relu_in, relu_out=relu_out, logits=False, skip_from=skip)


def _pool(c, hw):
    return dict(kind="maxpool", in_c=c, in_h=hw, in_w=hw, out_c=c, kh=3, kw=3, stride=2, pad=0,
                relu_in=False, relu_out=False, logits=False, skip_from=-1)


def _fc(k, n, relu_in=False, last=False):
    return dict(kind="fc", in_c=k, in_h=1, in_w=1, out_c=n, kh=1, kw=1, stride=1, pad=0,
                relu_in=relu_in, relu_out=not last, logits=last, skip_from=-1, value=False)


def _network(net, case):
    """(input kind, input shape, layers) of a case's network, one more column with a value head."""
    actions, value = case["actions"], case.get("value", False)
    if net == "mlp":
        dims = [case["obs"]] + [case["hidden"]] * 2
        layers = [_fc(dims[0], dims[1]), _fc(dims[1], dims[2])]
        shape, hidden = (case["obs"], 1, 1), case["hidden"]
    elif net in ("nature", "student"):
        c1, c2, c3, hidden = (32, 64, 64, 512) if net == "nature" else (16, 32, 32, 256)
        layers = [_conv(4, 84, c1, 8, 4, 0), _conv(c1, 20, c2, 4, 2, 0), _conv(c2, 9, c3, 3, 1, 0),
                  _fc(c3 * 49, hidden)]
        shape = FRAME
    else:
        layers, c, hw, hidden, shape = [], 4, 84, 256, FRAME
        for n in (16, 32, 32):
            layers += [_conv(c, hw, n, 3, 1, 1, relu_out=False), _pool(n, hw)]
            c, hw = n, (hw - 3) // 2 + 1
            for _ in range(2):
                x = len(layers) - 1
                layers += [_conv(c, hw, c, 3, 1, 1, relu_in=True),
                           _conv(c, hw, c, 3, 1, 1, relu_out=False, skip=x)]
        layers.append(_fc(c * hw * hw, hidden, relu_in=True))
    layers.append(_fc(hidden, actions + int(value), last=True))
    layers[-1]["value"] = value
    return ("f32" if net == "mlp" else "u8"), shape, layers


def _out_hw(l):
    return 1 if l["kind"] == "fc" else (l["in_h"] + 2 * l["pad"] - l["kh"]) // l["stride"] + 1


def _macs(layers):
    """Multiply-accumulates of one state."""
    return sum(_out_hw(l) ** 2 * l["out_c"] * l["in_c"] * l["kh"] * l["kw"]
               for l in layers if l["kind"] != "maxpool")


def _weights(layers):
    return sum(l["out_c"] * l["in_c"] * l["kh"] * l["kw"] for l in layers if l["kind"] != "maxpool")


# ------------------------------------------------------------------------------- inputs
def _int8_policy(net, case, rng):
    """An int8 policy with the weights and scales a calibrated network of this shape has: rounded
    normal weights (2:4 zeros in the residual network), scales that keep the second moment of a
    Kaiming ReLU network's activations."""
    kind, shape, layers = _network(net, case)
    m2 = 1.0 if net == "mlp" else 1.0 / 3.0
    s_input = np.float32((4.0 if net == "mlp" else 1.0) / 127.0)
    out, s = [], s_input
    for l in layers:
        e = dict(l, s_in=s, s_out=s, w=None, s_w=None, bias=None, skip_mul=None)
        if l["kind"] != "maxpool":
            n, c, k = l["out_c"], l["in_c"], l["kh"]
            w = np.clip(np.rint(rng.standard_normal((n, k, k, c), np.float32) * (127.0 / 4.0)), -127, 127)
            if net == "resnet":
                groups = w.reshape(n, -1, 4)
                order = np.argsort(rng.random(groups.shape, np.float32), axis=-1)
                np.put_along_axis(groups, order[..., :2], 0.0, axis=-1)
            e["w"] = np.ascontiguousarray(w.transpose(0, 3, 1, 2)).astype(np.int8)
            e["s_w"] = (4.0 * math.sqrt(2.0 / (c * k * k)) / 127.0 * rng.uniform(0.8, 1.2, n)).astype(np.float32)
            e["bias"] = (rng.standard_normal(n) * 0.01).astype(np.float32)
            if l["skip_from"] >= 0:
                m2 *= 2.0
                e["skip_mul"] = rng.integers(60, 200, n).astype(np.int32)
            e["s_out"] = np.float32(1.0 if l["logits"] else 5.0 * math.sqrt(2.0 * m2) / 127.0)
        out.append(e)
        s = e["s_out"]
    return dict(in_kind=kind, in_shape=shape, s_input=s_input, layers=out)


def _observations(net, case, batch, gen):
    if net == "mlp":
        return torch.randn((batch, case["obs"]), device="cuda", generator=gen)
    return torch.randint(0, 256, (batch,) + FRAME, dtype=torch.uint8, device="cuda", generator=gen)


def _generators(seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    return np.random.default_rng(seed), gen


def _outputs(batch, actions, **where):
    return (torch.empty((batch, actions), dtype=torch.float32, **where),
            torch.empty(batch, dtype=torch.int32, **where),
            torch.empty(batch, dtype=torch.float32, **where))


# ------------------------------------------------------------------------------- the cases
_CARTPOLE = dict(net="mlp", obs=4, hidden=64, actions=2)
_LUNAR = dict(net="mlp", obs=8, hidden=256, actions=4)


def listed():
    return [
        # an Actor on a classic-control task at the paper's batch of 160 environments: the smallest call
        dict(name="cartpole_b160", do="act", batch=160, **_CARTPOLE),
        # a wide vectorised gym Actor on vector observations
        dict(name="lunarlander_b4096", do="act", batch=4096, **_LUNAR),
        # the paper's own Actor step: Atari frames, original network, 160 environments
        dict(name="nature_b160", do="act", net="nature", actions=18, batch=160),
        # batched inference server for many Actors, original network
        dict(name="nature_b8192", do="act", net="nature", actions=18, batch=8192),
        # distilled student with the value and entropy outputs, a ragged number of environments
        dict(name="student_value_b1237", do="act_ex", net="student", actions=18, value=True, batch=1237),
        # the deep residual network for one Actor host
        dict(name="resnet_b100", do="act", net="resnet", actions=18, batch=100),
        # and for a large batched inference server
        dict(name="resnet_b16384", do="act", net="resnet", actions=18, batch=16384),
        # an Actor that steps its environments on the CPU: observations and results in host memory
        dict(name="host_nature_b160", do="host", net="nature", actions=18, batch=160),
        # linear-alpha strategy: each state follows the student with probability alpha
        dict(name="mixed_b2048", do="mixed", net="nature", actions=18, value=True, batch=2048, alpha=0.8),
        # an Actor beside a Learner that owns the free memory: fixed workspace, nothing allocated
        dict(name="noalloc_nature_b160", do="noalloc", net="nature", actions=18, batch=160),
        # Corrector and Monitor on a finished set of rollouts: V-trace targets and the KL indicators
        dict(name="rollout_16x8192", do="rollout", steps=16, batch=8192, actions=18, discounts=True),
        # the Compressor hands over new weights: quantise, calibrate, build the handle, first step, export
        dict(name="refresh_resnet", do="refresh", net="resnet", actions=18, rows=256, batch=160),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    do = rng.choice(["act", "act", "act", "act_ex", "host", "mixed", "noalloc", "rollout", "refresh"])
    if do == "rollout":
        return dict(do=do, steps=_log(rng, 5, 40), batch=_log(rng, 32, 6000), actions=rng.randint(2, 18),
                    discounts=rng.random() < 0.5)
    net = rng.choice(["mlp", "nature", "student", "resnet"] if do != "mixed" else ["nature"])
    case = dict(do=do, net=net, actions=rng.randint(3, 18))
    if net == "mlp":
        case.update(obs=rng.randint(3, 32), hidden=rng.choice([64, 128, 256]), actions=rng.randint(2, 8))
    if do == "act":
        case["batch"] = _log(rng, 1, 8192)
    elif do == "act_ex":
        case.update(batch=_log(rng, 1, 8192), value=True)
    elif do == "host":
        case["batch"] = _log(rng, 1, 8192)
    elif do == "mixed":
        case.update(batch=_log(rng, 1, 4096), value=rng.random() < 0.5, alpha=round(rng.uniform(0.1, 0.9), 2))
    elif do == "noalloc":  # bounded by the fixed workspace
        case["batch"] = _log(rng, 1, 150 if net == "resnet" else 1200)
    else:
        case.update(rows=_log(rng, 64, 200 if net == "resnet" else 1024), batch=_log(rng, 1, 512))
    return case


def prepare(case, seed):
    rng, gen = _generators(seed)
    do, batch = case["do"], case["batch"]
    s = dict(do=do, case=case)
    if do == "rollout":
        shape = (case["steps"], batch)
        logits = torch.randn((2,) + shape + (case["actions"],), device="cuda", generator=gen) * 2.0
        logits[1] = logits[0] + 0.3 * logits[1]  # the compressed policy follows the original one
        logp = torch.log_softmax(logits, dim=-1)
        taken = torch.multinomial(logp[1].exp().reshape(-1, case["actions"]), 1, generator=gen).reshape(shape + (1,))
        s["logits"] = [z.reshape(-1, case["actions"]).contiguous() for z in logits]
        s["logp"] = [z.gather(-1, taken).squeeze(-1).contiguous() for z in logp]
        s["rewards"] = torch.randint(-1, 2, shape, device="cuda", generator=gen).float()
        s["values"] = torch.randn(shape, device="cuda", generator=gen)
        s["bootstrap"] = torch.randn(batch, device="cuda", generator=gen)
        s["discounts"] = None
        if case["discounts"]:  # one episode in twenty steps ends
            s["discounts"] = 0.99 * (torch.rand(shape, device="cuda", generator=gen) > 0.05).float()
        return s
    net = case["net"]
    s["obs"] = _observations(net, case, batch, gen)
    s["u"] = torch.rand(batch, device="cuda", generator=gen)
    if do == "refresh":
        kind, shape, layers = _network(net, case)
        s["net"] = (kind, shape, layers)
        s["params"] = [None if l["kind"] == "maxpool" else dict(
            w=rng.standard_normal((l["out_c"], l["in_c"], l["kh"], l["kw"]), np.float32) *
            np.float32(math.sqrt(2.0 / (l["in_c"] * l["kh"] * l["kw"]))),
            bias=rng.standard_normal(l["out_c"], np.float32) * np.float32(0.01)) for l in layers]
        s["calib"] = _observations(net, case, case["rows"], gen).cpu().numpy()
        return s
    s["policy"] = P.Policy(_int8_policy(net, case, rng), 1 if do == "noalloc" else batch)
    if do == "mixed":
        s["small"] = P.Policy(_int8_policy("student", case, rng), batch)
        s["select"] = torch.rand(batch, device="cuda", generator=gen)
    elif do == "host":
        s["obs"], s["u"] = s["obs"].cpu().pin_memory(), s["u"].cpu().pin_memory()
        s["out"] = _outputs(batch, case["actions"], pin_memory=True)
    elif do == "noalloc":
        s["out"] = _outputs(batch, case["actions"], device="cuda")
    return s


def run(s):
    do, case = s["do"], s["case"]
    if do == "act":
        return s["policy"].act(s["obs"], s["u"])
    if do == "act_ex":
        return s["policy"].act_ex(s["obs"], s["u"])
    if do == "host":
        return s["policy"].act_host(s["obs"], s["u"], s["out"])
    if do == "mixed":
        return P.act_mixed(s["small"], s["policy"], s["obs"], s["u"], s["select"], case["alpha"])
    if do == "noalloc":
        out = s["out"]
        status = s["policy"].act_noalloc_raw(s["obs"].data_ptr(), s["u"].data_ptr(), case["batch"], out[0].data_ptr(),
                                             out[1].data_ptr(), out[2].data_ptr(),
                                             torch.cuda.current_stream().cuda_stream)
        if status:
            raise RuntimeError("act_noalloc: status %d" % status)
        return out
    if do == "rollout":
        targets = P.vtrace(s["logp"][1], s["logp"][0], s["rewards"], s["values"], s["bootstrap"], 0.99,
                           discounts=s["discounts"])
        return targets, P.kl(s["logits"][0], s["logits"][1])
    kind, shape, layers = s["net"]
    policy = P.Policy.from_fp32(kind, shape, layers, s["params"], s["calib"], case["batch"],
                                prune24=case["net"] == "resnet")
    first = policy.act(s["obs"], s["u"])
    exported = [policy.export(i) for i in range(len(layers))]
    policy.close()
    flat = {}
    for k in ("w", "s_w", "skip_mul"):  # one array of each for the whole network
        parts = [e[k].reshape(-1) for e in exported if e[k] is not None]
        if parts:
            flat[k] = np.concatenate(parts)
    flat["scales"] = np.array([[e["s_in"], e["s_out"]] for e in exported], np.float32)
    return first, flat


def work(case):
    batch, a = case["batch"], case["actions"]
    if case["do"] == "rollout":
        n = case["steps"] * batch
        vt = 4 * n * (7 if case["discounts"] else 6) + 4 * batch
        return dict(bytes=vt + n * (8 * a + 4) + 8, flops=n * (20 + 12 * a))
    kind, shape, layers = _network(case["net"], case)
    obs = int(np.prod(shape)) * (4 if kind == "f32" else 1)
    step_bytes = batch * (obs + 4 + 4 * a + 8 + (8 if case["do"] in ("act_ex", "mixed") else 0)) + _weights(layers)
    ops = 2.0 * batch * _macs(layers) / (2 if case["net"] == "resnet" and case["do"] != "refresh" else 1)
    if case["do"] == "mixed":  # a state needs the network it follows, not both
        small = _network("student", case)[2]
        return dict(bytes=step_bytes + _weights(small) + 5 * batch,
                    flops=2.0 * batch * (case["alpha"] * _macs(small) + (1 - case["alpha"]) * _macs(layers)))
    if case["do"] == "refresh":
        return dict(bytes=step_bytes + case["rows"] * obs + 5 * _weights(layers),
                    flops=ops + 2.0 * case["rows"] * _macs(layers))
    return dict(bytes=step_bytes, flops=ops)


def tolerance(case):
    """Logits, values, int8 weights and scales have one right bit pattern; log-probs, entropies, KL and
    V-trace targets are fp32 results of a few roundings; an action may differ where its uniform draw
    lies within rounding of a CDF edge."""
    if case["do"] == "rollout":
        return {"rel": 1e-5}
    return {"rel": 1e-5, "max": 1e-5, "differ": min(0.01, 2.0 / case["batch"])}
