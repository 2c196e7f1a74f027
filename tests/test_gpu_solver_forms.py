"""The two forms of the multigrid solvers (one cluster per component for the
whole solve, kernels per sweep on large systems) at the sizes where the
choice and the shape of the work change, against the Jacobi-preconditioned
solve (relaxation) and the persistent cooperative solve (pressure) of the same
systems."""
import pytest

import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1006_0720_gb300 as pg  # noqa: E402


def _relax(nx, ny, wall_tag=None):
    gm = pg.Mesh(inputs.channel_mesh(nx, ny, seed=4, wall_tag=wall_tag))
    gp = pg.Particles(gm, 3, ppe=30, u_sigma=0.1)
    p = pg.model_params(closure="glm")
    pg.pdf_estimate_stats(gp, gm)
    return gm, gp, p, torch.zeros((9, gm.n_nodes), dtype=torch.float64, device="cuda")


# unknowns: 6 x 11 = 66 (one level), 16 x 16 = 256 and 16 x 17 = 272 (one CTA, two),
# 32 x 64 and 32 x 65 = 2,048, 2,080 (the last size below and at eight CTAs),
# 64 x 128 = 8,192 (the largest of the cluster form) and 64 x 129
@pytest.mark.parametrize("nx,ny", [(7, 11), (17, 16), (17, 17), (33, 64), (33, 65), (65, 128), (65, 129)])
@pytest.mark.parametrize("wall_tag", [None, inputs.TAG_NOSLIP])
def test_relaxation_forms_agree_with_jacobi(nx, ny, wall_tag):
    """Both solves stop at a residual of 1e-12; the systems' condition keeps the
    solutions' difference below 1e3 times that."""
    gm, gp, p, wp = _relax(nx, ny, wall_tag)
    it, res = pg.pdf_relax_solve_particles(gp, gm, p, wp, rtol=1e-12, max_it=500)
    assert max(res) <= 1e-12
    pg.pdf_relax_set_solver(gp, False)
    ref = torch.zeros_like(wp)
    pg.pdf_relax_solve_particles(gp, gm, p, ref, rtol=1e-12, max_it=20000)
    scale = ref.abs().amax(dim=1, keepdim=True).clamp_min(1e-300)
    assert float(((wp - ref).abs() / scale).max()) < 1e-9


@pytest.mark.parametrize("nx,ny", [(17, 17), (65, 129)])
def test_relaxation_iteration_cap(nx, ny):
    """No, one and three iterations are too few: reported, and no more are made."""
    gm, gp, p, wp = _relax(nx, ny)
    for cap in (0, 1, 3):
        with pytest.raises(pg.PdfError) as e:
            pg.pdf_relax_solve_particles(gp, gm, p, wp.zero_(), rtol=1e-10, max_it=cap)
        assert e.value.status == pg.capi.PDF_ENOTCONV


# 20 x 40 - 40 = 760, 64 x 64 = 4,096 (the largest of the cluster form), 64 x 65
@pytest.mark.parametrize("nx,ny", [(9, 8), (17, 17), (20, 40), (65, 64), (65, 65)])
def test_pressure_forms_agree(nx, ny):
    """Residuals of 1e-12 on matrices of condition below 1e5."""
    m = inputs.channel_mesh(nx, ny, seed=2)
    out = []
    for persistent in (False, True):
        gm = pg.Mesh(m)
        gp = pg.Particles(gm, 5, ppe=30, u_sigma=0.2)
        p = pg.model_params(closure="glm", pressure="projection")
        pg.pdf_pressure_set_solver(gp, persistent)
        pg.pdf_estimate_stats(gp, gm)
        it, res = pg.pdf_pressure_project(gp, gm, p, rtol=1e-12, max_it=500)
        assert res <= 1e-12 and it <= 60
        out.append(pg.pdf_pressure_field(gp, gm))
    assert float((out[0] - out[1]).abs().max()) < 1e-7 * float(out[1].abs().max())
