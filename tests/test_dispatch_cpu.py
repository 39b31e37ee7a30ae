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
