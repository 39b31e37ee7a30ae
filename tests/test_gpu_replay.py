"""A network's forward pass from its second batch on is a graph replay: same logits as the calls one by one, for new
images, after a batch size change, after a plan change and inside a caller's own stream capture."""
from types import SimpleNamespace

import pytest
import torch

pytestmark = pytest.mark.gpu


def _net(seed=0):
    from paper_2003_07577_b200 import network
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    shapes = [("conv1", "first", 3, 16, 3, 1, 1, 16, 8), ("s1b1c1", "conv", 16, 16, 3, 1, 1, 16, 2),
              ("s1b1c2", "conv", 16, 16, 3, 1, 1, 16, 3), ("s2b1c1", "conv", 16, 32, 3, 2, 1, 16, 4),
              ("s2b1c2", "conv", 32, 32, 3, 1, 1, 8, 1), ("s2b1ds", "shortcut", 16, 32, 1, 2, 0, 16, 4),
              ("fc", "fc", 32, 10, 1, 1, 0, 1, 8)]
    layers = [SimpleNamespace(name=n, role=r, c_in=ci, c_out=co, k=k, stride=s, pad=p, h_in=h, w_in=h, w_bits=3, a_bits=a,
                              w_scale=0.05) for n, r, ci, co, k, s, p, h, a in shapes]
    codes = {L.name: torch.randint(-4, 4, (L.c_out, L.c_in, L.k, L.k), generator=g, device="cuda", dtype=torch.int8)
             for L in layers}
    return network.BasicBlockNet(network.calibrated_plans(layers, codes, _images(4, g))), g


def _images(n, g):
    return torch.randint(0, 256, (n, 16, 16, 3), generator=g, device="cuda", dtype=torch.uint8)


def _one_by_one(net, x):
    """The reference: a fresh object's first pass, which issues the calls themselves."""
    from paper_2003_07577_b200 import network
    fresh = network.BasicBlockNet(net.plans)
    return fresh.forward(x).clone()


def test_replayed_batches_equal_the_calls_one_by_one():
    net, g = _net()
    for n in (3, 3, 3, 1, 1, 1, 3):                      # recording at the second batch of a size, replay from there
        x = _images(n, g)
        assert torch.equal(net.forward(x), _one_by_one(net, x))
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    got = net.forward(x, stream=side)
    torch.cuda.synchronize()
    assert torch.equal(got, _one_by_one(net, x))


def test_replay_follows_plan_changes():
    net, g = _net(1)
    x = _images(2, g)
    for _ in range(3):
        before = net.forward(x).clone()
    net.plans[1].ch_bias = net.plans[1].ch_bias + 1.0
    for _ in range(3):
        after = net.forward(x).clone()
        assert torch.equal(after, _one_by_one(net, x)) and not torch.equal(after, before)
    net.plans[-1].desc.a_scale *= 2.0                    # a field of a descriptor, changed in place
    assert torch.equal(net.forward(x), _one_by_one(net, x)) and not torch.equal(net.forward(x), after)


def test_forward_inside_a_callers_capture():
    net, g = _net(2)
    x = _images(2, g)
    for _ in range(3):
        want = net.forward(x).clone()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        out = net.forward(x)
    out.zero_()
    graph.replay()
    assert torch.equal(out, want)


def test_replay_follows_pooling_and_storage_changes():
    """What the calls read when they are issued: the pooling, the plan objects, the storage behind a weight tensor."""
    from paper_2003_07577_b200 import network
    net, g = _net(3)
    x = _images(2, g)
    want = [net.forward(x).clone() for _ in range(3)][-1]

    w = net.plans[1].packed_w                            # other storage behind the same tensor object
    kept = w.data
    w.data = torch.zeros_like(w)
    zeroed = net.forward(x).clone()
    assert torch.equal(zeroed, _one_by_one(net, x)) and not torch.equal(zeroed, want)
    w.data = kept
    assert torch.equal(net.forward(x), want)

    import copy
    other = copy.copy(net.fc)                            # another plan object in the place of one
    other.ch_bias = other.ch_bias + 1.0
    mine, net.fc = net.fc, other
    shifted = net.forward(x).clone()
    assert torch.allclose(shifted, want + 1.0)
    net.fc = mine
    assert torch.equal(net.forward(x), want)


def test_replay_follows_an_assigned_pooling():
    """The maximum pooling after the first convolution of an ImageNet network, changed on the object: window and padding, so
    that the sizes behind it stay."""
    from paper_2003_07577_b200 import network
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    shapes = [("conv1", "first", 3, 16, 3, 2, 1, 32, 8), ("s1b1c1", "conv", 16, 16, 3, 1, 1, 8, 2),
              ("s1b1c2", "conv", 16, 16, 3, 1, 1, 8, 3), ("fc", "fc", 16, 10, 1, 1, 0, 1, 8)]
    layers = [SimpleNamespace(name=n, role=r, c_in=ci, c_out=co, k=k, stride=s, pad=p, h_in=h, w_in=h, w_bits=3, a_bits=a,
                              w_scale=0.05) for n, r, ci, co, k, s, p, h, a in shapes]
    codes = {L.name: torch.randint(-4, 4, (L.c_out, L.c_in, L.k, L.k), generator=g, device="cuda", dtype=torch.int8) for L in layers}
    x = torch.randint(0, 256, (2, 32, 32, 3), generator=g, device="cuda", dtype=torch.uint8)
    plans = network.calibrated_plans(layers, codes, x, pool=(3, 2, 1))
    net = network.BasicBlockNet(plans, pool=(3, 2, 1))
    before = [net.forward(x).clone() for _ in range(3)][-1]
    net.pool = (2, 2, 0)
    after = [net.forward(x).clone() for _ in range(3)]
    want = network.BasicBlockNet(plans, pool=(2, 2, 0)).forward(x)
    assert all(torch.equal(a, want) for a in after) and not torch.equal(want, before)
