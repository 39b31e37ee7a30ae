"""The tile kernel's per-tap form (family "umma" where no strip fits: wide images, strides above 2, more than 64 taps) and the
library's own choice for such layers against the CPU oracle: every activation bitwidth, ragged channels and pixel tiles, split
reductions, every output and shortcut form, weight levels."""
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


CASES = [
    # n, c, co, (kh, kw), (sh, sw), (ph, pw), h, w, ab, levels
    (1, 64, 64, (3, 3), (1, 1), (1, 1), 3, 224, 4, 0),        # a tap row is 226 pixels of frame
    (2, 45, 77, (3, 3), (1, 1), (1, 1), 2, 200, 5, 0),        # ragged channels, tiles and images
    (1, 64, 48, (3, 3), (1, 1), (1, 1), 2, 210, 2, 0),
    (1, 33, 64, (5, 5), (1, 1), (2, 2), 4, 97, 3, 0),
    (2, 64, 64, (3, 3), (3, 3), (1, 1), 29, 31, 1, 0),
    (1, 100, 130, (4, 4), (4, 4), (0, 0), 16, 20, 8, 0),
    (3, 512, 40, (1, 1), (3, 3), (0, 0), 9, 8, 6, 0),
    (1, 256, 64, (3, 3), (3, 3), (1, 1), 7, 7, 7, 0),         # 72 reduction words on one pixel tile: split over a cluster
    (1, 64, 64, (3, 3), (4, 4), (1, 1), 1, 1, 4, 0),          # a single output pixel, one tap inside
    (1, 3, 64, (11, 11), (4, 4), (2, 2), 40, 44, 8, 0),       # 121 taps of one word
    (2, 40, 96, (9, 9), (1, 1), (4, 4), 8, 9, 2, 0),          # 81 taps of two words
    (1, 70, 64, (1, 17), (1, 3), (0, 20), 5, 33, 3, 0),       # one row of taps, padding wider than the taps' reach
    (1, 64, 64, (3, 3), (3, 1), (1, 1), 12, 20, 4, 1),        # weight levels: the window sum as an accumulator column
    (1, 96, 40, (5, 5), (1, 1), (2, 2), 2, 100, 2, 1),
    (1, 640, 40, (3, 3), (3, 3), (1, 1), 6, 6, 2, 1),         # weight levels with a split reduction
]


@pytest.mark.parametrize("shortcut", ["none", "fp32", "packed"])
@pytest.mark.parametrize("case", CASES)
def test_tap_form(ebs, U, oracle, case, shortcut):
    n, c, co, (kh, kw), s, pad, h, w, ab, levels = case
    rng = np.random.default_rng(n + c + co + kh + kw + h + w + ab)
    wb, nb = 3, 5
    qa = U.rand_codes(rng, (n, c, h, w), ab, False)
    qw = rng.integers(-3, 4, size=(co, c, kh, kw), dtype=np.int32)
    d = ebs.conv_desc(c, co, kh, kw, *s, *pad, wb, ab, 0.02, 0.05, levels)
    acc = (oracle.conv2d_levels if levels else oracle.conv2d_codes)(qa, qw, s, pad)
    S = oracle.combined_scale(0.02, 0.05)
    cs, cb = rng.uniform(0.5, 2.0, co).astype(np.float32), rng.uniform(-0.3, 0.3, co).astype(np.float32)
    to = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(U.dev())  # noqa: E731
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
    assert ran >= 5                                           # the choice and the tiles of 32 channels and more
    assert ebs.ebs_device_wait_timeouts() == 0


def test_library_choice_without_packing(ebs, U, oracle):
    """32-bit results alone, where the choice lies between the tile kernel and the warp-level kernels."""
    for n, c, co, k, s, h, w, b in [(1, 16, 48, 3, 1, 4, 200, 4), (1, 64, 64, 3, 1, 48, 200, 2), (1, 64, 96, 3, 1, 5, 200, 3),
                                    (1, 3, 64, 3, 1, 4, 200, 2), (1, 3, 64, 3, 1, 4, 200, 6), (2, 64, 64, 3, 3, 20, 20, 2),
                                    (1, 64, 64, 3, 1, 32, 32, 2), (2, 20, 50, 3, 1, 9, 11, 5), (3, 33, 16, 3, 1, 7, 7, 8),
                                    (2, 30, 40, 5, 1, 9, 9, 3), (2, 16, 32, 3, 2, 13, 12, 4)]:
        rng = np.random.default_rng(c + co + h)
        qa, qw = U.rand_codes(rng, (n, c, h, w), b, False), U.rand_codes(rng, (co, c, k, k), b, True)
        d = U.desc_for(c, co, k, s, 1, b, b)
        assert np.array_equal(U.run_conv(qa, qw, d)["acc"], oracle.conv2d_codes(qa, qw, (s, s), (1, 1))), (c, co, s)
    for n, c, co, s, h, w, b in [(1, 64, 64, 1, 32, 32, 4), (2, 100, 129, 2, 9, 8, 3), (3, 33, 10, 1, 5, 7, 8)]:      # 1x1
        rng = np.random.default_rng(c + co + h)
        qa, qw = U.rand_codes(rng, (n, c, h, w), b, False), U.rand_codes(rng, (co, c, 1, 1), b, True)
        d = U.desc_for(c, co, 1, s, 0, b, b)
        assert np.array_equal(U.run_conv(qa, qw, d)["acc"], oracle.conv2d_codes(qa, qw, (s, s), (0, 0))), (c, co, s)
