"""Frame transforms at the largest second extents (the grid's limit of blocks along y) and over the
range of values.

The analysis is compared with the oracle: three passes of at most three roundings each with taps of absolute
sum <= 1. Scaling the values and the threshold by a power of two scales the result by it, bit for bit,
as long as no square of a coefficient passes FP32's range (1.8e19); without a threshold, up to its end."""
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


def scaled(shape, k):
    f = torch.randn(shape, device="cuda", generator=torch.Generator(device="cuda").manual_seed(6))
    return f, f * 2.0**k


@pytest.mark.parametrize("k, mu", [(-40, 1.5), (56, 1.5), (60, 1.5), (122, 0.0)])
def test_range_of_the_fused_step(cb, k, mu):
    f, g = scaled((9, 31, 37), k)
    out = cb.tf_shrink(f, mu, False)
    assert mu == 0.0 or not torch.allclose(out, f, rtol=0.1)  # the threshold takes effect
    assert torch.equal(cb.tf_shrink(g, mu * 2.0**k, False), out * 2.0**k)


# 38 and 37 columns: the kernels for one position per lane and, in 16 bits, for a pair
@pytest.mark.parametrize("nx", [37, 38])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("k, mu", [(-40, 3.0), (60, 3.0), (122, 0.0)])
def test_range_of_the_synthesis(cb, k, mu, dtype, nx):
    a, b = (v.to(dtype) for v in scaled((27, 9, 31, nx), k))
    out = cb.tf_synthesize_shrink(a, mu, False)
    assert torch.equal(cb.tf_synthesize_shrink(b, mu * 2.0**k, False), out * 2.0**k)


# widths about a warp (32 and 34 columns), and FP32 rows of whole sectors that leave a pair tile half empty (72, 96)
# or not (104, 160), each beside the next even width: both kernels agree bit for bit
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("nx", [32, 34, 72, 74, 96, 98, 104, 160, 162])
def test_analysis_widths(cb, nx, dtype):
    shape = (5, 13, nx)
    f = torch.randn(shape, device="cuda", generator=torch.Generator(device="cuda").manual_seed(7))
    a = cb.tf_analyze(f, dtype=dtype)
    single = torch.empty(a.numel() + 1, dtype=dtype, device="cuda")[1:].view(a.shape)
    assert torch.equal(a, cb.tf_analyze(f, out=single))
    ref = oracle.tf_analyze(f.cpu().numpy())
    eps = 0.0 if dtype == torch.float32 else 2.0**-8
    err = np.abs(a.float().cpu().numpy() - ref)
    assert np.all(err <= 10 * 2.0**-24 * float(f.abs().max()) + eps * np.abs(ref) * 1.001 + 2.0**-25)


# blocks of 12 warps (20 rows; 256x256x8 leaves blocks of 16 warps a third of the SMs idle) and of 16 warps (28 rows):
# whole tiles, one row and one column more, the z-fastest order of a thin volume
@pytest.mark.parametrize("shape", [(1, 20, 28), (5, 21, 29), (30, 40, 57), (8, 256, 256), (40, 84, 128), (40, 85, 127), (128, 128, 18), (120, 130, 33)])
def test_fused_step_block_sizes(cb, shape):
    f = np.random.default_rng(8).standard_normal(shape).astype(np.float32)
    out = cb.tf_shrink(torch.from_numpy(f).cuda(), 1.5, False).cpu().numpy()
    ref = oracle.tf_synthesize(oracle.tf_shrink(oracle.tf_analyze(f), 1.5))
    assert np.linalg.norm(out - ref) <= 1e-5 * np.linalg.norm(ref)
