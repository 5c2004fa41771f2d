"""Float32 patch applies of a batch: patches of the class blocks against the
same patches with a block each, and the lane counts against each other."""
import numpy as np
import pytest

from paper_2403_11636_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fc():
    from paper_2403_11636_gb300 import fc as m
    return m


# a chunk and less, ragged last chunks, levels of one chunk, more than one
# grid shape in a batch
BATCHES = {
    "2d": lambda: [inputs.channel_2d(0, n=8, nlevels=2), inputs.channel_2d(1, n=48, nlevels=3),
                   inputs.channel_2d(2, n=208, nlevels=5)],
    "3d": lambda: [inputs.channel_3d(0, n=8, nlevels=2), inputs.channel_3d(1, n=24, nlevels=3)],
}


def cycle(fc, probs, prec, dedup, tile):
    import torch
    B = fc.Batch([fc.Solver(p, prec=prec, dedup=dedup) for p in probs], tile=tile)
    b = torch.as_tensor(inputs.uniform_array(int(B.ndof), 3)).cuda()
    x = torch.zeros_like(b)
    B.vcycle_(x, b)
    out = x.cpu().numpy()
    B.close()
    return out


@pytest.mark.parametrize("prec", ["fp32", "bf16"])
@pytest.mark.parametrize("name", list(BATCHES))
def test_class_patches_and_lane_counts(fc, name, prec):
    """A patch adds in the same order with a shared and with its own block, so
    the two agree bit for bit.  Another lane count is another order: 402
    products in float32, whose magnitudes add up to about 100 times the update
    (alpha-scaled rows), 402 * 6e-8 * 100 = 2.4e-3 in the worst case and its
    root, 1.2e-4, at random; 1e-3."""
    probs = BATCHES[name]()
    ref = None
    for tile in [(1, 128, 4), (2, 512, 2), (4, 256, 4), (8, 128, 16), (16, 512, 2), (32, 128, 2), (32, 256, 8),
                 (32, 512, 1)]:
        got = cycle(fc, probs, prec, 1, tile)
        np.testing.assert_array_equal(got, cycle(fc, probs, prec, 0, tile), err_msg=str(tile))
        assert np.all(np.isfinite(got))
        if ref is None:
            ref = got
        assert np.max(np.abs(got - ref)) <= 1e-3 * np.max(np.abs(ref)), tile
