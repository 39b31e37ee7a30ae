"""The tile kernel (family "umma": 128 pixels x a channel tile, reduction split over a cluster) against the CPU oracle at the
edges of its rules: ragged words per cluster rank, one pixel, partial channel tiles, every output and shortcut form, weight
levels, strides, and layers beyond the warp-level kernels' tap tables."""


import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ebs():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2003_07577_b200 import binding
    binding.lib()
    return binding


@pytest.fixture(scope="module")
def U(ebs):
    from tests import _util
    return _util


@pytest.mark.parametrize("shortcut", ["none", "fp32", "packed"])
@pytest.mark.parametrize("case", [
    # n, c, co, k, stride, pad, h, w, ab, levels
    (1, 288, 64, 3, 1, 1, 5, 5, 4, 0),       # nine words over a cluster of eight would leave ranks empty: fewer ranks
    (1, 512, 96, 3, 1, 1, 7, 7, 3, 0),       # deep reduction on one pixel tile: eight ranks
    (2, 1024, 130, 1, 1, 0, 3, 3, 8, 0),     # partial channel tile and word
    (1, 4096, 33, 1, 1, 0, 1, 1, 1, 0),      # a single output pixel
    (3, 96, 64, 3, 2, 1, 13, 12, 5, 0),      # four phase images
    (9, 64, 128, 3, 1, 1, 7, 7, 2, 0),       # images across a pixel tile, no split
    (2, 200, 70, 3, 1, 1, 6, 5, 6, 1),       # weight levels: the window sum as an accumulator column
    (1, 640, 40, 3, 1, 1, 6, 6, 2, 1),       # weight levels with a split reduction
    (1, 1024, 64, 5, 1, 2, 6, 6, 2, 0),      # 800 reduction words
])
def test_tile_kernel_edges(ebs, U, oracle, case, shortcut):
    n, c, co, k, s, pad, h, w, ab, levels = case
    rng = np.random.default_rng(sum(case))
    wb, nb = 3, 5
    qa = U.rand_codes(rng, (n, c, h, w), ab, False)
    qw = rng.integers(-3, 4, size=(co, c, k, k), dtype=np.int32)
    d = ebs.conv_desc(c, co, k, k, s, s, pad, pad, wb, ab, 0.02, 0.05, levels)
    acc = oracle.conv2d_levels(qa, qw, (s, s), (pad, pad)) if levels else oracle.conv2d_codes(qa, qw, (s, s), (pad, pad))
    S = oracle.combined_scale(0.02, 0.05)
    cs, cb = rng.uniform(0.5, 2.0, co).astype(np.float32), rng.uniform(-0.3, 0.3, co).astype(np.float32)
    to = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(U.dev())
    res, extra = None, {}
    if shortcut == "fp32":
        res = rng.standard_normal(acc.shape).astype(np.float32)
        extra = dict(residual=to(res.transpose(0, 2, 3, 1)))
    elif shortcut == "packed":
        q_res = U.rand_codes(rng, acc.shape, 3, False)
        res = oracle.dequant_codes(q_res, 0.11)
        extra = dict(res_packed=U.pack_acts_codes(q_res, 3), res_bits=3, res_scale=0.11)
    y0, _ = oracle.epilogue(acc, S, cs, cb, res, relu=True)
    step = np.float32(max(float(np.percentile(y0, 98)), 1e-3) / ((1 << nb) - 1))
    y_ref, q_ref = oracle.epilogue(acc, S, cs, cb, res, relu=True, next_bits=nb, inv_next=np.float32(1.0) / step)
    epi = ebs.epilogue(to(cs), to(cb), extra.pop("residual", None), True, nb, float(step), **extra)
    px, pw = U.pack_acts_codes(qa, ab), U.pack_weight_codes(qw, d)
    ran = 0
    for variant in [-1] + U.variants_of("umma"):
        if variant >= 0 and not U.applies(d, h, w, variant, n=n, epi=epi, want_y=True, want_packed=True):
            continue
        out = U.run_conv(qa, qw, d, epi, want_acc=True, want_y=True, next_bits=nb, variant=variant, px=px, pw=pw)
        assert np.array_equal(out["acc"], acc), f"variant {variant}: accumulators"
        assert np.array_equal(out["y"], y_ref), f"variant {variant}: fp32 outputs"
        assert np.array_equal(out["packed"], oracle.pack_acts(q_ref, nb)), f"variant {variant}: packed words"
        out = U.run_conv(qa, qw, d, epi, want_acc=False, next_bits=nb, variant=variant, px=px, pw=pw)
        assert np.array_equal(out["packed"], oracle.pack_acts(q_ref, nb)), f"variant {variant}: packed only"
        ran += 1
    assert ran >= 4
    assert ebs.ebs_device_wait_timeouts() == 0


def test_tile_kernel_chain_of_dependent_launches(ebs, U, oracle):
    """Twelve layers back to back, each reading the one before: a launch begins before its predecessor has ended, its first
    read must still see the predecessor's planes."""
    rng = np.random.default_rng(3)
    d = U.desc_for(128, 128, 3, 1, 1, 3, 4, 0.03, 0.07)
    qw = rng.integers(-3, 4, size=(128, 128, 3, 3), dtype=np.int32)
    q = U.rand_codes(rng, (2, 128, 14, 14), 4, False)
    S = oracle.combined_scale(0.03, 0.07)
    pw, px = U.pack_weight_codes(qw, d), U.pack_acts_codes(q, 4)
    want, epis = [], []
    for _ in range(12):
        acc = oracle.conv2d_codes(q, qw, (1, 1), (1, 1))
        y0, _ = oracle.epilogue(acc, S, relu=True)
        step = np.float32(np.percentile(y0, 99) / 15)
        _, q = oracle.epilogue(acc, S, relu=True, next_bits=4, inv_next=np.float32(1.0) / step)
        assert 0 < q.mean() < 15
        want.append(oracle.pack_acts(q, 4))
        epis.append(ebs.epilogue(relu=True, next_a_bits=4, next_a_scale=float(step)))
    bufs = [px] + [torch.empty_like(px) for _ in range(12)]
    for i in range(12):
        ebs.ebs_conv2d_mixed(bufs[i], 2, 14, 14, pw, d, epis[i], None, None, bufs[i + 1])
    torch.cuda.synchronize()
    for i in range(12):
        assert np.array_equal(U.as_u32(bufs[i + 1]).reshape(2, 14, 14, 4, 4), want[i]), f"layer {i}"
