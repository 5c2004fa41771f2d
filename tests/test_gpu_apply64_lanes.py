"""FC_APPLY64_TPP sets the lanes of the FP64 patch apply on levels with class
products too: the sums of the nodes that these leave change their order, and
agree to rounding."""
import os
import subprocess
import sys

import numpy as np
import pytest

from tests.gpu_util import rel

pytestmark = pytest.mark.gpu

RUN = """
import sys, numpy as np
from paper_2403_11636_gb300 import fc, inputs
p = inputs.porous_3d(3, n=64, nspheres=12, nlevels=5)
x = inputs.random_vector(p, 5)
np.save(sys.argv[1], fc.Solver(p).smooth(x, inputs.random_vector(p, 6)).cpu().numpy() - x)
"""


def test_lanes_on_a_level_with_class_products(tmp_path):
    out = {}
    for lanes in (4, 8, 16, 32):
        f = str(tmp_path / f"{lanes}.npy")
        subprocess.run([sys.executable, "-c", RUN, f], check=True, env={**os.environ, "FC_APPLY64_TPP": str(lanes)})
        out[lanes] = np.load(f)
    for lanes in (4, 16, 32):
        assert rel(out[lanes], out[8]) <= 1e-11      # as in test_gpu_digits.py
        assert np.count_nonzero(out[lanes] != out[8]) > len(out[8]) // 10
