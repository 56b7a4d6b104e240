"""Imagers at the widths where counts pass 32 bits: rows of the adjoint's prefix table of 2 GiB (2^28
columns), and nearly 2^31 columns, which the allocation-free projection takes in batches.

The volume's shadow lies in the first 41 columns, which a narrow imager repeats; every other column
misses it. The adjoint's bar is the operators' relative L2 of 1e-4 against the FP64 oracle on the
narrow imager; the projections run the same sums in the same order and are equal."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

U_FIRST, NARROW, WIDE = -19.75, 41, 1 << 28


def geom(nu, nv=3):
    return synth.Geometry(nx=7, ny=5, nz=6, dx=1.0, dy=1.1, dz=1.2, nu=nu, nv=nv, du=1.0, dv=2.3, v_off=0.4, n_views=1,
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


def test_static_projection_of_nearly_2_31_columns():
    import paper_1008_2042_gb300 as cb

    cb.load_library()
    if torch.cuda.mem_get_info()[0] < 72 << 30:
        pytest.skip("needs 63 GB of device memory")
    g, nu = geom(NARROW, nv=1), 2**31 - 2
    f = torch.tensor(synth.random_volume(g, 84), dtype=torch.float32, device="cuda")
    with cb.Geometry(g) as h:
        p = cb.project(h, f)
    assert int(torch.count_nonzero(p)) >= 5
    with cb.Geometry(geom(nu, nv=1)) as h:
        q = torch.full((1, 1, nu), float("nan"), dtype=torch.float32, device="cuda")
        cb.project_static(h, f, q)
    assert torch.equal(p, q[:, :, :NARROW])
    assert int(torch.count_nonzero(q[:, :, NARROW:])) == 0
