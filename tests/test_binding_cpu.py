"""The Python entry points' checks of their arguments, without a device: what a kernel could not read
raises before anything is launched (a null handle stands in for the policy: a call that gets past the
checks ends in the library's own error instead)."""
import ctypes as C

import numpy as np
import pytest

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def P():
    from paper_2211_15023_b200 import build
    build.build()
    import paper_2211_15023_b200 as package
    return package


def _policy(P, in_kind="f32"):
    g = P.Policy.__new__(P.Policy)
    g._h, g._raw = C.c_void_p(), 0
    g.in_kind, g.in_shape, g.n_actions, g.value_head, g.max_batch = in_kind, (4, 1, 1), 2, False, 16
    return g


def test_tensors_the_device_cannot_read_raise_before_the_launch(P):
    g, obs, u = _policy(P), torch.zeros((16, 4)), torch.zeros(16)
    x, boot = torch.zeros((3, 16)), torch.zeros(16)
    for call in (lambda: g.act_ex(obs, u), lambda: g.act_ex(obs.double(), u),
                 lambda: P.act_mixed(g, g, obs, u, u, 0.5), lambda: P.kl(obs, obs),
                 lambda: P.vtrace(x, x, x, x, boot, 0.99)):
        with pytest.raises(AssertionError):
            call()
