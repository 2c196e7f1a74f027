"""The projection with the inflow/outflow condition where much of the mesh is
inflow and outflow: those unknowns never coarsen, so the coarsest system is
large (up to all unknowns, without a single level).  The kernels per sweep and
the persistent cooperative solve give the same field."""
import numpy as np
import pytest

import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1006_0720_gb300 as pg  # noqa: E402


def _strip(ny):
    """One column of cells between inflow and outflow: every node is on one of the two."""
    y = np.linspace(-1.0, 1.0, ny)
    period = 2.0 * (y[1] - y[0])
    j = np.arange(ny - 1)
    a, b, c, d = 2 * j, 2 * j + 1, 2 * j + 3, 2 * j + 2  # counter-clockwise
    tri = np.concatenate([np.stack([a, b, c], 1), np.stack([a, c, d], 1)]).astype(np.int32)
    bnd = [(0, 1, inputs.TAG_WALL), (2 * ny - 2, 2 * ny - 1, inputs.TAG_WALL)]
    bnd += [(2 * k, 2 * k + 2, inputs.TAG_INFLOW) for k in j] + [(2 * k + 1, 2 * k + 3, inputs.TAG_OUTFLOW) for k in j]
    twin = np.arange(2 * ny) ^ 1
    return dict(xy=np.stack([np.tile([0.0, period], ny), np.repeat(y, 2)], 1), tri=tri, bnd=np.asarray(bnd, dtype=np.int32),
                twin=twin.astype(np.int32), period=float(period))


# unknowns, those of inflow and outflow: 180, 120 (the coarsest system just below the
# cluster form's limit); 300, 200; 2,100, 1,400; 128, 3,200 and 4,200: all of them
@pytest.mark.parametrize("nx,ny", [(3, 60), (3, 100), (3, 700), (2, 64), (2, 1600), (2, 2100)])
def test_open_boundary_forms_agree(nx, ny):
    m = _strip(ny) if nx == 2 else inputs.channel_mesh(nx, ny, seed=2, inout=True)
    out = []
    for persistent in (False, True):
        gm = pg.Mesh(m)
        gp = pg.Particles(gm, 5, ppe=30, u_sigma=0.2)
        p = pg.model_params(closure="glm", Pi=0.5, pressure="projection_inout")
        pg.pdf_pressure_set_solver(gp, persistent)
        pg.pdf_estimate_stats(gp, gm)
        it, res = pg.pdf_pressure_project(gp, gm, p, rtol=1e-12, max_it=500)
        assert res <= 1e-12 and it <= 60
        out.append(pg.pdf_pressure_field(gp, gm))
    assert float((out[0] - out[1]).abs().max()) < 1e-7 * float(out[1].abs().max())
