"""V-cycles and solves on the default streams, whose coarse part is recorded on
a stream of the handle and replayed, give the same bits as on a stream of the
caller's, as with profiling, which launches every kernel by itself."""
from types import SimpleNamespace

import numpy as np
import pytest

from paper_2403_11636_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fc():
    from paper_2403_11636_gb300 import fc as m
    return m


KINDS = {
    "fp64": (inputs.channel_2d(0, n=64, nlevels=4), {}),
    "fp64 3d": (inputs.porous_3d(3, n=16, nspheres=6, nlevels=3), {}),
    "matrix 3d": (inputs.porous_3d(3, n=16, nspheres=6, nlevels=3), {"cache": "matrix"}),
    "pairs": (inputs.porous_3d(3, n=16, nspheres=6, nlevels=3), {"prec": "df64"}),
    "fp32": (inputs.channel_2d(0, n=64, nlevels=4), {"prec": "fp32"}),
    "q2": (inputs.channel_2d(0, n=32, nlevels=3), {"element": "q2"}),
}


@pytest.mark.parametrize("kind", list(KINDS))
def test_default_streams(fc, kind):
    import torch
    p, opt = KINDS[kind]
    out = {}
    # the handles 1 and 2 name the default streams (torch knows the first only;
    # its own copies run on that, which waits for the second)
    for name, ptr in (("own", None), ("null", 0), ("legacy", 1), ("thread", 2)):
        stream = torch.cuda.Stream() if ptr is None else SimpleNamespace(cuda_stream=ptr)
        torch.cuda.synchronize()
        with torch.cuda.stream(stream if ptr is None else torch.cuda.default_stream()):
            s = fc.Solver(p, stream=stream, **opt)
            x, b = inputs.uniform_array(s.ndof(), 5), inputs.uniform_array(s.ndof(), 7)
            got = [s.vcycle(x, b), s.vcycle(x, b)]          # recorded, replayed
            s.profile(True)
            got.append(s.vcycle(x, b))
            s.profile(False)
            got.append(s.solve(s.rhs(), rtol=1e-6)[0])
            s.sync()
            out[name] = [v.cpu().numpy() for v in got]
            s.close()
    for name, got in out.items():
        for k, v in enumerate(got):
            np.testing.assert_array_equal(v, out["own"][k], err_msg=f"{name} {k}")
        np.testing.assert_array_equal(got[0], got[1])
        np.testing.assert_array_equal(got[0], got[2])
