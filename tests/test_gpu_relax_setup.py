"""The relaxation multigrid's matrices as they are formed on the device: systems
that are nothing but the coarsest matrix (its inverse is the whole
preconditioner) and one whose finest products take one thread per entry,
against the Jacobi-preconditioned solve."""
import pytest

import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1006_0720_gb300 as pg  # noqa: E402


# unknowns 2 x 3, 3 x 3, 4 x 6 = 24 (300 entries of the triangle: two rounds of 256
# threads), 7 x 9 = 63, 8 x 8 = 64 (the largest); 128 x 160 = 20,480.  The inverse is
# exact to FP32 rounding (2^-24 times a condition of at most 1e4): each iteration
# gains a factor of a thousand or more, six reach 1e-12, two more for the
# FP32 product.
@pytest.mark.parametrize("nx,ny,most", [(3, 3, 8), (4, 3, 8), (5, 6, 8), (8, 9, 8), (9, 8, 8), (129, 160, 60)])
@pytest.mark.parametrize("wall_tag", [None, inputs.TAG_NOSLIP])
def test_multigrid_matrices(nx, ny, most, wall_tag):
    gm = pg.Mesh(inputs.channel_mesh(nx, ny, seed=4, wall_tag=wall_tag))
    gp = pg.Particles(gm, 3, ppe=30, u_sigma=0.1)
    p = pg.model_params(closure="glm")
    pg.pdf_estimate_stats(gp, gm)
    wp, ref = (torch.zeros((9, gm.n_nodes), dtype=torch.float64, device="cuda") for _ in range(2))
    it, res = pg.pdf_relax_solve_particles(gp, gm, p, wp, rtol=1e-12, max_it=500)
    assert max(res) <= 1e-12
    assert max(it) <= most
    pg.pdf_relax_set_solver(gp, False)
    pg.pdf_relax_solve_particles(gp, gm, p, ref, rtol=1e-12, max_it=20000)
    scale = ref.abs().amax(dim=1, keepdim=True).clamp_min(1e-300)
    assert float(((wp - ref).abs() / scale).max()) < 1e-9
