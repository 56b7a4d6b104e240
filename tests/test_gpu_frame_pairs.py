"""The frame transforms' kernels for pairs of adjacent positions against the general ones.

An even contiguous extent and aligned arrays take two positions per lane; arrays that start
off a pair's alignment, and odd extents, take one. Both use the same operations in the same order,
so that they agree bit for bit; the analysis is also compared with the oracle.
"""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu

# (nz, ny, nx): one and two planes, odd rows, tiles of 64 x 4 (analysis) and 60 x 14 (synthesis) missed by a pair
SHAPES = [(1, 1, 2), (2, 3, 4), (3, 5, 62), (5, 13, 64), (4, 15, 66), (7, 4, 122), (9, 17, 130)]


@pytest.fixture(scope="module")
def cb():
    import paper_1008_2042_gb300 as m

    m.load_library()
    return m


def off_by_one(shape, dtype):
    n = int(np.prod(shape))
    return torch.empty(n + 1, dtype=dtype, device="cuda")[1:].view(shape)


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16, torch.float16])
@pytest.mark.parametrize("shape", SHAPES)
def test_analysis_pairs(cb, shape, dtype):
    f = np.random.default_rng(3).standard_normal(shape).astype(np.float32)
    fd = torch.from_numpy(f).cuda()
    pair = cb.tf_analyze(fd, dtype=dtype)
    single = cb.tf_analyze(fd, out=off_by_one((27,) + shape, dtype))
    assert torch.equal(pair, single)
    # three passes of at most three roundings each, taps of absolute sum <= 1; then one rounding to the type
    eps = {torch.float32: 0.0, torch.bfloat16: 2.0**-8, torch.float16: 2.0**-11}[dtype]
    ref = oracle.tf_analyze(f)
    err = np.abs(pair.float().cpu().numpy() - ref)
    assert np.all(err <= 10 * 2.0**-24 * np.abs(f).max() + eps * np.abs(ref) * 1.001 + 2.0**-25)


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float16])
@pytest.mark.parametrize("shape", SHAPES)
def test_synthesis_pairs(cb, shape, dtype):
    rng = np.random.default_rng(4)
    pair = torch.from_numpy(rng.standard_normal((27,) + shape).astype(np.float32)).cuda().to(dtype)
    single = off_by_one((27,) + shape, dtype)
    single.copy_(pair)
    assert torch.equal(cb.tf_synthesize_shrink(pair, 3.0, False), cb.tf_synthesize_shrink(single, 3.0, False))
