"""Frame transforms at the largest second extents (the grid's limit of blocks along y).

The analysis is compared with the oracle: three passes of at
most three roundings each with taps of absolute sum <= 1."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def cb():
    import paper_1008_2042_gb300 as m

    m.load_library()
    return m


# the last extent of the pair kernel's tiles of 4 rows, the first beyond it, the last that is accepted
@pytest.mark.parametrize("ny", [262140, 262141, 524280])
def test_analysis_of_tall_planes(cb, ny):
    f = np.random.default_rng(5).standard_normal((1, ny, 2)).astype(np.float32)
    a = cb.tf_analyze(torch.from_numpy(f).cuda()).cpu().numpy()
    assert np.abs(a - oracle.tf_analyze(f)).max() <= 10 * 2.0**-24 * np.abs(f).max()
