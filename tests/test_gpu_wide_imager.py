"""The adjoint on an imager whose rows of the prefix table are 2 GiB long (2^28 columns).

The volume's shadow lies in the first 41 columns, which a narrow imager repeats; every other column
misses it, so its ones have no part in the result. Bar: the operators' relative L2 of 1e-4 against
the FP64 oracle on the narrow imager."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

U_FIRST, NARROW, WIDE = -19.7, 41, 1 << 28


def geom(nu):
    return synth.Geometry(nx=7, ny=5, nz=6, dx=1.0, dy=1.1, dz=1.2, nu=nu, nv=3, du=1.0, dv=2.3, v_off=0.4, n_views=1,
                          u_off=U_FIRST + 0.5 * (nu - 1), angles=(0.3,))


def test_backproject_with_table_rows_of_2_gib():
    import paper_1008_2042_gb300 as cb

    cb.load_library()
    if torch.cuda.mem_get_info()[0] < 24 << 30:
        pytest.skip("needs 20 GB of device memory")
    g = geom(NARROW)
    y = synth.random_projections(g, 83)
    ref = oracle.backproject(g, y)
    assert np.count_nonzero(ref) >= 100
    wide = torch.ones((1, g.nv, WIDE), dtype=torch.float32, device="cuda")
    wide[:, :, :NARROW] = torch.tensor(y, dtype=torch.float32, device="cuda")
    with cb.Geometry(geom(WIDE)) as h:
        b = cb.backproject(h, wide).cpu().numpy()
    assert np.linalg.norm(b - ref) <= 1e-4 * np.linalg.norm(ref)
