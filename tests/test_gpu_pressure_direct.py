"""Pressure systems of at most 256 unknowns: the dense inverse is the whole
preconditioner, with either condition at the ends."""
import pytest

import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1006_0720_gb300 as pg  # noqa: E402


# unknowns: 9 x 8 = 72, 16 x 16 = 256, 9 x 28 = 252 of which 56 are open, 16 x 16 with 32.
# FP64 inverses of condition below 1e5: the first iteration leaves a residual of
# 1e-16 x 1e5 x 10, one more is allowed
@pytest.mark.parametrize("nx,ny,inout", [(10, 8, False), (17, 16, False), (9, 28, True), (16, 16, True)])
def test_small_systems_are_solved_directly(nx, ny, inout):
    gm = pg.Mesh(inputs.channel_mesh(nx, ny, seed=2, inout=inout))
    gp = pg.Particles(gm, 5, ppe=30, u_sigma=0.2)
    p = pg.model_params(closure="glm", Pi=0.5, pressure="projection_inout" if inout else "projection")
    pg.pdf_estimate_stats(gp, gm)
    it, res = pg.pdf_pressure_project(gp, gm, p, rtol=1e-10, max_it=100)
    assert res <= 1e-10 and it <= 2
