"""The polynomials of the mixed form's non-nearest Ewald images (csrc/common.cuh,
erfc_image_p0 / p1): the source's coefficients are the committed fit, and their
FP32 evaluation gives erfc(sqrt y)/sqrt y and its derivative to 1e-6 on the range
of y that kappa L between the kernel's limits reaches (the fit's 4e-7 plus a few
FP32 roundings)."""
import os
import re

import numpy as np
import pytest

pytest.importorskip("scipy")
from paper_1605_08423_gb300 import fit_erfc

SRC = open(os.path.join(os.path.dirname(fit_erfc.__file__), "csrc", "common.cuh")).read()


def _coefficients(which):
    body = SRC[SRC.index(f"float erfc_image_p{which}(float t)"):]
    body = body[:body.index("return p;")]
    hi = float(re.search(r"float p = ([-\d.e+]+)f;", body).group(1))
    rest = [float(v) * (1.0 if sg == "+" else -1.0) for sg, v in re.findall(r"p \* t ([-+]) ([\d.e+-]+)f;", body)]
    return np.array(list(reversed([hi] + rest)))


@pytest.mark.parametrize("which", [0, 1])
def test_source_is_the_fit(which):
    c = _coefficients(which)
    assert len(c) == fit_erfc.IMAGE_DEGREES[which] + 1
    assert np.allclose(c, fit_erfc.fit_image(which), rtol=2e-7, atol=1e-9)


@pytest.mark.parametrize("which", [0, 1])
def test_fp32_accuracy(which):
    lo, hi = (float(re.search(name + r" = ([\d.]+)f", SRC).group(1)) for name in ("kImageKLMin", "kImageKLMax"))
    y_lo, y_hi = lo ** 2 / 4, 0.64 * hi ** 2          # r from L/2 to the cutoff 0.8 L
    assert y_lo >= fit_erfc.Y_MIN and y_hi <= fit_erfc.Y_MAX
    y = np.linspace(y_lo, y_hi, 20001)
    t = (1.0 / y).astype(np.float32)
    p = np.float32(0)
    for c in _coefficients(which)[::-1].astype(np.float32):
        p = (p * t + c).astype(np.float32)
    got = (p * t).astype(np.float64)
    assert np.max(np.abs(got / fit_erfc.image_target(which, y) - 1.0)) < 1e-6
