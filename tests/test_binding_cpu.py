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


def test_act_noalloc_raw_takes_every_kind_of_address_and_number_ctypes_takes(P):
    """Integers, None, ctypes pointers, numpy integers for the batch; what is none of these raises."""
    g, INVALID = _policy(P), 1
    buf = (C.c_float * 4)()
    for args in ((0, 0, 5, 0, 0, 0), (None, None, 5, None, None, None, None), (0, 0, np.int64(5), 0, 0, 0),
                 (C.c_void_p(0), None, 5, buf, C.byref(buf), 0, C.c_void_p(0)), (0, 0, np.int32(5), 0, 0, 0),
                 (0, 0, True, 0, 0, 0), (0, 0, 1 << 70, 0, 0, 0), (0, 0, -1, 0, 0, 0)):
        assert g.act_noalloc_raw(*args) == INVALID, args
    for args in ((0, 0, 5.0, 0, 0, 0), (0, 0, None, 0, 0, 0), (0, 0, "5", 0, 0, 0), (2.0, 0, 5, 0, 0, 0)):
        with pytest.raises(C.ArgumentError):
            g.act_noalloc_raw(*args)
