"""The give-up path of the bounded device-side waits (collected after the other kernel tests: it raises the
library's give-up counter, which those tests expect to be zero)."""
import os

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ebs():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import paper_2003_07577_b200 as pkg
    from paper_2003_07577_b200 import binding
    if not os.path.exists(binding.LIB_PATH):
        pkg.build()
    binding.lib()
    return binding


@pytest.fixture(scope="module")
def U(ebs):
    from tests import _util
    return _util


@pytest.mark.parametrize("form", ["single", "pair"])
def test_pipe_bounded_waits_give_up_and_recover(ebs, U, oracle, form):
    """The give-up path, made to run on purpose without faulting anything: with the wait limit at a few polls and the
    issuing thread told to issue no tensor-core work, every wait for the tensor core runs out with nothing in flight;
    each thread block raises its abort flag, leaves its loops, frees its tensor memory and returns.  The counter rises,
    ebs_check_device_status reports EBS_ERR_TIMEOUT once, and the next healthy launch is bit-exact."""
    rng = np.random.default_rng(5)
    qa = U.rand_codes(rng, (4, 64, 12, 12), 3, False)
    co = 64 if form == "single" else 256                      # the pair of CTAs works on whole 256-channel tiles
    qw = U.rand_codes(rng, (co, 64, 3, 3), 2, True)
    d = U.desc_for(64, co, 3, 1, 1, 2, 3)
    ref = oracle.conv2d_codes(qa, qw, (1, 1), (1, 1))
    variant = U.variants_of("umma_pipe")[0 if form == "single" else -1]
    assert U.applies(d, 12, 12, variant, n=4)
    assert ebs.ebs_check_device_status() == ebs.EBS_OK
    before = ebs.ebs_device_wait_timeouts()
    ebs.ebs_test_set_device_wait(64, True)
    try:
        U.run_conv(qa, qw, d, variant=variant)              # returns: every wait is bounded
    finally:
        ebs.ebs_test_set_device_wait(0, False)
    after = ebs.ebs_device_wait_timeouts()
    assert after > before, "no thread block reported that it gave up"
    assert ebs.ebs_check_device_status() == ebs.EBS_ERR_TIMEOUT
    assert ebs.ebs_check_device_status() == ebs.EBS_OK        # reported once
    got = U.run_conv(qa, qw, d, variant=variant)["acc"]       # the context is healthy: same launch, exact result
    assert np.array_equal(got, ref)
    assert ebs.ebs_device_wait_timeouts() == after


@pytest.mark.parametrize("limit", [1, 64])
@pytest.mark.parametrize("co", [64, 256])
def test_pipe_gives_up_with_tensor_copies_in_flight(ebs, U, oracle, co, limit):
    """Packed words by tensor copies: the copies of the next slots are under way when the expanders' waits run out (for a free stage,
    and with a single poll for the words themselves).  Whole warps leave their loops, the block drains its copies and returns."""
    rng = np.random.default_rng(co + limit)
    qa, qw = U.rand_codes(rng, (2, 1024, 40, 37), 6, False), U.rand_codes(rng, (co, 1024, 1, 1), 2, True)
    d = U.desc_for(1024, co, 1, 1, 0, 2, 6)
    variant = U.variants_of("umma_pipe")[0 if co == 64 else 2]
    route = ebs.ebs_test_conv_route(d, 2, 40, 37, variant=variant)
    assert route["tensor_copies"] and route["stage_words"] * route["stages"] < 32      # more words than the stages hold
    px, pw = U.pack_acts_codes(qa, 6), U.pack_weight_codes(qw, d)
    assert ebs.ebs_check_device_status() == ebs.EBS_OK
    before = ebs.ebs_device_wait_timeouts()
    ebs.ebs_test_set_device_wait(limit, 1)
    try:
        U.run_conv(qa, qw, d, variant=variant, px=px, pw=pw)                            # returns: every wait is bounded
    finally:
        ebs.ebs_test_set_device_wait(0, 0)
    after = ebs.ebs_device_wait_timeouts()
    assert after > before, "no thread block reported that it gave up"
    assert ebs.ebs_check_device_status() == ebs.EBS_ERR_TIMEOUT
    got = U.run_conv(qa, qw, d, variant=variant, px=px, pw=pw)["acc"]
    assert np.array_equal(got, oracle.conv2d_codes(qa, qw, (1, 1), (0, 0)))
    assert ebs.ebs_device_wait_timeouts() == after


def test_tile_kernel_does_not_count_the_launch_before_it(ebs, U, oracle):
    """A tile launch may start while the one before it runs; what it waits for then is not a stage that never fills.  The second
    launch's limit (2000 polls, 80 us and more) covers its own 10 us many times, but not the first launch's: 2304 MMAs of 104
    clocks on one accumulator, 0.12 ms, queued four times."""
    rng = np.random.default_rng(11)
    slow = U.desc_for(8192, 256, 3, 1, 1, 1, 1)
    qs, ws = np.ones((1, 8192, 2, 2), dtype=np.int32), U.rand_codes(rng, (256, 8192, 3, 3), 1, True)
    d = U.desc_for(64, 64, 3, 1, 1, 2, 3)
    qa, qw = U.rand_codes(rng, (1, 64, 8, 8), 3, False), U.rand_codes(rng, (64, 64, 3, 3), 2, True)
    px, pw, pxs, pws = U.pack_acts_codes(qa, 3), U.pack_weight_codes(qw, d), U.pack_acts_codes(qs, 1), U.pack_weight_codes(ws, slow)
    wide, narrow = U.variants_of("umma")[-1], U.variants_of("umma")[2]
    acc = torch.empty((1, 2, 2, 256), dtype=torch.int32, device=U.dev())
    out = torch.empty((1, 8, 8, 64), dtype=torch.int32, device=U.dev())
    before = ebs.ebs_device_wait_timeouts()
    for _ in range(3):                                       # (first calls load code)
        out.zero_()
        for _ in range(4):
            ebs.ebs_conv2d_mixed(pxs, 1, 2, 2, pws, slow, None, acc, None, None, variant=wide)
        ebs.ebs_test_set_device_wait(2000, False)
        try:
            ebs.ebs_conv2d_mixed(px, 1, 8, 8, pw, d, None, out, None, None, variant=narrow)
        finally:
            ebs.ebs_test_set_device_wait(0, False)
        torch.cuda.synchronize()
        assert ebs.ebs_device_wait_timeouts() == before
        assert np.array_equal(out.cpu().numpy().transpose(0, 3, 1, 2), oracle.conv2d_codes(qa, qw, (1, 1), (1, 1)))


@pytest.mark.parametrize("c,hw,limit,skip", [
    (64, 12, 64, 1),            # one thread block per tile
    (512, 7, 64, 1),            # a cluster per tile, every member gives up before the exchange of the sums
    (512, 7, 4000, 2),          # ... in the exchange: one member's sums never come
    (64, 300, 64, 1),           # per-tap form (a row of 300 pixels)
])
def test_tile_bounded_waits_give_up_and_recover(ebs, U, oracle, c, hw, limit, skip):
    rng = np.random.default_rng(c + hw)
    h, w = (3, hw) if hw > 100 else (hw, hw)
    qa, qw = U.rand_codes(rng, (1, c, h, w), 3, False), U.rand_codes(rng, (64, c, 3, 3), 2, True)
    d = U.desc_for(c, 64, 3, 1, 1, 2, 3)
    variant = U.variants_of("umma")[2]
    assert ebs.ebs_check_device_status() == ebs.EBS_OK
    before = ebs.ebs_device_wait_timeouts()
    ebs.ebs_test_set_device_wait(limit, skip)
    try:
        U.run_conv(qa, qw, d, variant=variant)              # returns: every wait is bounded
    finally:
        ebs.ebs_test_set_device_wait(0, 0)
    after = ebs.ebs_device_wait_timeouts()
    assert after > before, "no thread block reported that it gave up"
    assert ebs.ebs_check_device_status() == ebs.EBS_ERR_TIMEOUT
    got = U.run_conv(qa, qw, d, variant=variant)["acc"]
    assert np.array_equal(got, oracle.conv2d_codes(qa, qw, (1, 1), (1, 1)))
    assert ebs.ebs_device_wait_timeouts() == after


def test_whole_network_bounded_waits_give_up_and_recover(ebs):
    from types import SimpleNamespace
    from paper_2003_07577_b200 import network
    g = torch.Generator(device="cuda")
    g.manual_seed(7)
    shapes = [("conv1", "first", 3, 16, 3, 1, 1, 16, 8), ("s1b1c1", "conv", 16, 16, 3, 1, 1, 16, 2),
              ("s1b1c2", "conv", 16, 16, 3, 1, 1, 16, 3), ("s2b1c1", "conv", 16, 32, 3, 2, 1, 16, 4),
              ("s2b1c2", "conv", 32, 32, 3, 1, 1, 8, 1), ("s2b1ds", "shortcut", 16, 32, 1, 2, 0, 16, 4),
              ("fc", "fc", 32, 10, 1, 1, 0, 1, 8)]
    layers = [SimpleNamespace(name=n, role=r, c_in=ci, c_out=co, k=k, stride=s, pad=p, h_in=h, w_in=h, w_bits=3, a_bits=a,
                              w_scale=0.05) for n, r, ci, co, k, s, p, h, a in shapes]
    codes = {L.name: torch.randint(-4, 4, (L.c_out, L.c_in, L.k, L.k), generator=g, device="cuda", dtype=torch.int8) for L in layers}
    x = torch.randint(0, 256, (3, 16, 16, 3), generator=g, device="cuda", dtype=torch.uint8)
    plans = network.calibrated_plans(layers, codes, x)
    want = network.BasicBlockNet(plans).forward(x).clone()
    net = network.FusedBasicBlockNet(plans)
    before = ebs.ebs_device_wait_timeouts()
    ebs.ebs_test_set_device_wait(64, 1)
    try:
        net.forward(x)
        torch.cuda.synchronize()
    finally:
        ebs.ebs_test_set_device_wait(0, 0)
    assert ebs.ebs_device_wait_timeouts() == before + 3       # one thread block an image
    assert ebs.ebs_check_device_status() == ebs.EBS_ERR_TIMEOUT
    assert torch.equal(net.forward(x), want)
    assert ebs.ebs_device_wait_timeouts() == before + 3
