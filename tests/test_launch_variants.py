"""Register-cap variants of the wave kernels that the autotuner tries: those that
are the same code as variant 0 are skipped, and only those."""
import ctypes as ct

import pytest

TRACE, SHADE, SHADOW, REVERSE = range(4)
BSDF, NEE, GUIDED, LIGHT = 1, 2, 4, 8


@pytest.mark.parametrize("tech", [BSDF, BSDF | NEE, BSDF | NEE | GUIDED, BSDF | NEE | LIGHT, BSDF | LIGHT])
def test_only_equal_variants_are_skipped(tech):
    from paper_2410_20429_gb300 import build as B
    lib = ct.CDLL(B.build())
    # bool mars::wave_variant_repeats(int kernel, int variant, int techniques)
    repeats = lib._ZN4mars20wave_variant_repeatsEiii
    repeats.restype = ct.c_bool
    for k in (TRACE, SHADE, SHADOW, REVERSE):
        # the light connection kernels are launched in the shadow kernel's variant
        own_code = k == REVERSE or (k == SHADOW and tech & LIGHT)
        assert [repeats(k, v, tech) for v in range(3)] == [False, not own_code, False]
