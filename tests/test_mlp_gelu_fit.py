"""The polynomial of the inference kernel's GELU (CPU): with the constants as
the source gives them, t exp(-t^2/2) P(1/(1 + k t)) stays within 3.3e-9 of
t erfc(t/sqrt 2)/2 for every t >= 0."""
import os
import re

import numpy as np
from scipy.special import erfc

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2512_12934_gb300", "csrc",
                   "lbm_mlp.cu")


def test_fit_error_of_the_packed_gelu():
    text = open(SRC).read()
    body = text[text.index("float2 gelu2(float2 z)"):]
    c = [float(v) for v in re.findall(r"(-?\d\.\d+)f", re.search(r"float c\[7\] = \{(.*?)\}", body, re.S)[1])]
    k = float(re.search(r"make_float2\((0\.\d+)f, 0\.\d+f\), make_float2\(1\.f", body)[1])
    assert len(c) == 7
    t = np.concatenate([np.linspace(0.0, 14.0, 400001), np.geomspace(14.0, 1e4, 2001)])
    exact = 0.5 * t * erfc(t / np.sqrt(2.0))
    for cast in (float, np.float32):  # as written, and as the kernel holds them
        u, p = 1.0 / (1.0 + float(cast(k)) * t), np.zeros_like(t)
        for a in c[::-1]:
            p = p * u + float(cast(a))
        assert np.abs(-t * np.exp(-0.5 * t * t) * p - exact).max() < 3.3e-9
