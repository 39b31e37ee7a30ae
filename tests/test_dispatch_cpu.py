"""Which kernel families the library offers for a layer (host-side rules; nothing is launched, no GPU needed)."""
import os

import pytest


@pytest.fixture(scope="module")
def ebs():
    import paper_2003_07577_b200 as pkg
    from paper_2003_07577_b200 import binding
    if not os.path.exists(binding.LIB_PATH):
        pkg.build()
    binding.lib()
    return binding


@pytest.mark.parametrize("c,co,k,stride,h,w", [
    (64, 64, 3, 1, 224, 224),          # tap rows further apart than a strip holds
    (64, 64, 5, 1, 96, 96),
    (64, 128, 7, 1, 64, 64),
    (64, 128, 3, 3, 112, 112),         # strides without phase images
    (96, 64, 4, 4, 112, 112),
    (256, 96, 1, 4, 160, 160),
    (64, 64, 9, 1, 28, 28),            # more taps than the tables of the strip forms
    (3, 64, 11, 4, 224, 224),
    (512, 512, 3, 3, 28, 28),
])
@pytest.mark.parametrize("levels", [0, 1])
def test_wide_and_strided_layers_have_a_tcgen05_kernel(ebs, c, co, k, stride, h, w, levels):
    d = ebs.conv_desc(c, co, k, k, stride, stride, k // 2, k // 2, 4, 4, 0.05, 0.05, levels)
    fams = [ebs.ebs_conv_variant_family(v) for v in range(ebs.ebs_num_conv_variants())
            if ebs.ebs_conv_variant_applies(d, 2, h, w, None, True, False, False, v) == ebs.EBS_OK]
    assert fams.count("umma") == 5, sorted(set(fams))


def _route(ebs, n, h, w, c, co, k, stride, ab, nb, terms=False, tile=None):
    """Route of a layer whose result is packed planes (stand-in buffers: nothing is read)."""
    d = ebs.conv_desc(c, co, k, k, stride, stride, k // 2, k // 2, 4, ab, 0.05, 0.05)
    epi = ebs.epilogue(None, None, None, True, nb, 1.0)
    if terms:
        epi.ch_scale_dev = epi.ch_bias_dev = 256
    pipe = [v for v in range(ebs.ebs_num_conv_variants()) if ebs.ebs_conv_variant_family(v) == "umma_pipe"]
    variant = -1 if tile is None else pipe[{64: 0, 128: 1, 256: 2, "pair": 3}[tile]]
    return ebs.ebs_test_conv_route(d, n, h, w, epi, False, False, True, variant)


@pytest.mark.parametrize("layer,tile,terms,want", [
    # n, h, w, c, co, k, stride, planes in, planes out
    ((256, 28, 28, 512, 256, 1, 1, 7, 7), 256, False, dict(pass_words=4, tensor_copies=1, resident=1)),
    ((256, 7, 7, 512, 2048, 1, 1, 7, 6), 256, False, dict(pass_words=4, tensor_copies=1, resident=1)),
    ((256, 28, 28, 512, 128, 1, 1, 5, 4), 128, False, dict(pass_words=2, tensor_copies=1, resident=1)),
    ((256, 56, 56, 256, 128, 1, 1, 7, 7), 128, False, dict(pass_words=2, tensor_copies=1, resident=1)),
    ((256, 28, 28, 128, 128, 3, 1, 7, 7), 128, True, dict(resident=1)),
    ((64, 28, 28, 128, 128, 3, 1, 7, 7), 128, True, dict(resident=1, pass_words=2)),
    ((64, 56, 56, 128, 128, 3, 2, 7, 5), 128, True, dict(resident=1, pass_words=3)),
    ((2, 83, 84, 64, 1024, 3, 1, 7, 5), 256, False, dict(resident=1)),
    ((4, 110, 55, 1280, 128, 1, 2, 6, 4), 128, True, dict(pass_words=4)),
    ((256, 58, 29, 608, 2048, 1, 2, 5, 7), 256, False, dict(pass_words=4)),
])
def test_ring_of_packed_words_displaces_neither_weights_nor_words(ebs, layer, tile, terms, want):
    """Where shared memory is short the ring of packed words is two slots deep, so that the words of an expander pass, resident weights of
    a k x k layer and tensor copies are what they are beside any ring (wide plane counts with rows of planes on their way out)."""
    got = _route(ebs, *layer, terms=terms, tile=tile)
    assert {k: got[k] for k in want} == want, got
    assert got["raw_slots"] >= 2 and got["stages"] >= 2


@pytest.mark.parametrize("layer", [
    (1, 67, 182, 256, 1280, 3, 1, 4, 4), (1, 136, 105, 1792, 768, 3, 1, 6, 5), (1, 24, 112, 1984, 256, 3, 1, 3, 4), (1, 138, 57, 192, 256, 3, 1, 7, 5),
    (1, 95, 41, 1280, 256, 1, 1, 8, 4),
])
def test_pair_of_thread_blocks_takes_streamed_layers(ebs, layer):
    """Streamed weights beside the widest stages: three slots of the weight ring are made room for."""
    got = _route(ebs, *layer, tile="pair")
    assert got["weight_slots"] >= 3 and got["stages"] >= 2, got


@pytest.mark.parametrize("layer,family", [
    # n, h, w, c, co, k, stride, planes in, planes out; the faster family as measured (rounds of 128 x 128 tiles on 148 SMs)
    ((4, 86, 86, 608, 64, 1, 1, 7, 7), "umma"), ((4, 115, 115, 544, 64, 1, 1, 7, 2), "umma"),          # no tensor copies: 1.6 and 2.8 rounds
    ((4, 77, 78, 1056, 128, 1, 1, 5, 4), "umma"), ((4, 60, 60, 288, 256, 1, 1, 5, 4), "umma"),         # 1.3, 1.5
    ((4, 115, 115, 64, 64, 1, 1, 7, 4), "umma"), ((4, 80, 81, 160, 256, 1, 1, 7, 7), "umma_pipe"),     # 2.8, 2.7
    ((4, 54, 54, 256, 256, 1, 1, 6, 2), "umma"), ((4, 43, 43, 256, 512, 1, 1, 5, 7), "umma_pipe"),     # tensor copies: 1.2, 1.6
    ((4, 71, 72, 512, 256, 1, 1, 5, 7), "umma_pipe"), ((16, 28, 28, 512, 128, 1, 1, 7, 4), "umma_pipe"),   # 2.2, 0.7
])
def test_layers_of_5_to_7_planes_run_on_the_faster_kernel(ebs, layer, family):
    got = _route(ebs, *layer)
    assert ebs.ebs_conv_variant_family(got["variant"]) == family, got
