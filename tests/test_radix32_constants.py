"""The FP32 constants of the radix-32 butterflies (turn32 in csrc/fft.cuh): each pair (c, r) stands for the turn
c + i c r by 2 pi k / 32.  The error in length is what a forward and an inverse line do not cancel; rounded each
by itself, c and r leave up to 3.04e-8."""
import math
import os
import re

import numpy as np

FFT = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1408_1782_gb300", "csrc",
                   "fft.cuh")


def _errors(c, r, k):
    z = complex(c, c * r) * complex(math.cos(math.pi * k / 16), -math.sin(math.pi * k / 16))
    return abs(z) - 1.0, z.imag


def _neighbours(x):
    x = np.float32(x)
    up, down = np.nextafter(x, np.float32(9e9)), np.nextafter(x, np.float32(-9e9))
    return [float(v) for v in (np.nextafter(down, np.float32(-9e9)), down, x, up, np.nextafter(up, np.float32(9e9)))]


def test_turns_are_the_nearest_to_length_one():
    text = open(FFT).read()
    pairs = re.findall(r"Turn\{(0x[0-9a-f.p+-]+)f, (0x[0-9a-f.p+-]+)f\}", text[text.index("turn32(int k)"):])
    assert len(pairs) == 7
    for k, (c, r) in enumerate(pairs, start=1):
        c, r = float.fromhex(c), float.fromhex(r)
        assert c == float(np.float32(c)) and r == float(np.float32(r))
        length, angle = _errors(c, r, k)
        assert abs(length) < 2.5e-8 and abs(angle) < 6.0e-8
        cost = [abs(a) + 0.05 * abs(b) for a, b in
                (_errors(x, y, k) for x in _neighbours(math.cos(math.pi * k / 16))
                 for y in _neighbours(math.tan(math.pi * k / 16)))]
        assert abs(length) + 0.05 * abs(angle) <= min(cost) * (1 + 1e-6) + 1e-15
