"""Argument checks of the CPython extension: what ctypes refused for these calls is refused, before the library is reached."""
import ctypes
import importlib.util
import os

import numpy as np
import pytest
import torch


@pytest.fixture()
def fast():
    """A module of its own (not the one the binding uses), with streams that need no GPU."""
    import paper_2003_07577_b200 as pkg
    from paper_2003_07577_b200 import binding as ebs
    pkg.build()
    L = ebs.lib()
    path = os.path.join(os.path.dirname(ebs.__file__), "_fastcall.so")
    spec = importlib.util.spec_from_file_location("_fastcall", path)
    m = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(m)
    names = ("ebs_pack_acts", "ebs_pack_acts_s2d", "ebs_conv2d_mixed", "ebs_conv2d_mixed_variant", "ebs_dequant",
             "ebs_global_avgpool", "ebs_maxpool_packed", "ebs_resnet_cifar_forward", "ebs_search_weight_forward",
             "ebs_search_act_forward", "ebs_graph_launch")
    m.bind({k: ctypes.cast(getattr(L, k), ctypes.c_void_p).value for k in names}, lambda device: 0, lambda: 0,
           ebs.ebs_conv_desc, ebs.ebs_epilogue, ebs.ebs_fused_head)
    yield m
    ebs._fast = None                                       # the extension's state is per process: the binding binds anew


def _pack(bits):
    return (None, 1, 1, 1, 8, 4, 4, bits, 1.0, None, None)


@pytest.mark.parametrize("bad", [2.7, "5", None, np.float32(2), torch.tensor(2.0)])
def test_integers_are_not_converted(fast, bad):
    with pytest.raises(TypeError):
        fast.pack_acts(*_pack(bad))
    with pytest.raises(TypeError):
        fast.global_avgpool(None, bad, 1, 1, None, None)
    with pytest.raises(TypeError):
        fast.dequant(None, bad, 8, 1.0, None, None, False, None, None)
    with pytest.raises(OverflowError):
        fast.pack_acts(*_pack(1 << 32))


@pytest.mark.parametrize("good", [2, True, np.int64(2), np.uint8(2), torch.tensor(2)])
def test_integer_types_are_taken(fast, good):
    from paper_2003_07577_b200 import binding as ebs
    assert fast.pack_acts(*_pack(good)) == ebs.EBS_ERR_INVALID_ARG       # (no buffers)
    assert fast.dequant(None, good, 8, 1.0, None, None, False, None, None) == ebs.EBS_ERR_INVALID_ARG


def test_structures_have_their_type(fast):
    from paper_2003_07577_b200 import binding as ebs
    d = ebs.conv_desc(8, 8, 1, 1, 1, 1, 0, 0, 2, 2, 0.1, 0.1)
    e = ebs.epilogue(None, None, None, True)
    call = lambda d, e: fast.conv2d_mixed(None, 1, 4, 4, None, d, e, None, None, None, None, -1)  # noqa: E731
    assert call(d, None) == call(d, e) == ebs.EBS_ERR_INVALID_ARG        # reaches the library, which misses its buffers
    for bad_d, bad_e in [(None, None), (bytes(d), None), (e, None), (d, bytes(e)), (d, d), (bytearray(ctypes.sizeof(d)), None)]:
        with pytest.raises(TypeError):
            call(bad_d, bad_e)
    head = lambda h, stride=0: fast.resnet_cifar_forward(None, 1, 8, 8, None, 1, h, None, None, stride, None)  # noqa: E731
    assert head(ebs.ebs_fused_head()) == ebs.EBS_ERR_INVALID_ARG
    for bad in (None, bytes(ctypes.sizeof(ebs.ebs_fused_head)), d):
        with pytest.raises(TypeError):
            head(bad)
    with pytest.raises(TypeError):
        head(ebs.ebs_fused_head(), 0.5)


def test_candidates_are_what_int_and_float_take(fast):
    from paper_2003_07577_b200 import binding as ebs
    call = lambda b, c: fast.search_act_forward(None, 16, 1.0, b, c, None, None)  # noqa: E731
    for bits, coeff in [([1, 2], [0.5, 0.5]), (np.array([1, 2]), np.array([0.5, 0.5])), ((1.0, "2"), ("0.5", 1)),
                        (torch.tensor([1, 2]), torch.tensor([0.5, 0.5]))]:
        assert call(bits, coeff) == ebs.EBS_ERR_INVALID_ARG
    for bits, coeff in [(3, [1.0]), ((b for b in (1, 2)), [0.5, 0.5]), ([None], [1.0]), ([1], ["x"]), ([1, 2], [1.0])]:
        with pytest.raises((TypeError, ValueError)):
            call(bits, coeff)
