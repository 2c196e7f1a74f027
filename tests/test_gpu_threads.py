"""Solves of different sizes from several host threads at once, each with its own
handles and stream: none disturbs another."""
import threading

import pytest

import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1006_0720_gb300 as pg  # noqa: E402


def _relaxation(nx, ny, max_it=500):
    gm = pg.Mesh(inputs.channel_mesh(nx, ny, seed=4))
    gp = pg.Particles(gm, 3, ppe=30, u_sigma=0.1)
    pg.pdf_estimate_stats(gp, gm)
    p = pg.model_params(closure="glm")
    wp = torch.zeros((9, gm.n_nodes), dtype=torch.float64, device="cuda")

    def solve():
        pg.pdf_relax_solve_particles(gp, gm, p, wp.zero_(), rtol=1e-12, max_it=max_it)
        return wp.clone()
    return solve


def _projection(nx, ny, max_it=500):
    gm = pg.Mesh(inputs.channel_mesh(nx, ny, seed=4))
    gp = pg.Particles(gm, 3, ppe=30, u_sigma=0.1)
    p = pg.model_params(closure="glm", pressure="projection")
    zero = torch.zeros(gm.n_nodes, dtype=torch.float64, device="cuda")
    st = {k: v.clone() for k, v in gp.get_state().items()}

    def solve():
        gp.set_state(st)
        pg.pdf_estimate_stats(gp, gm)
        pg.pdf_pressure_field(gp, gm, set=zero)
        pg.pdf_pressure_project(gp, gm, p, rtol=1e-10, max_it=max_it)
        return pg.pdf_pressure_field(gp, gm)
    return solve


# the largest cluster forms (8,192 and 4,096 unknowns) beside six threads with
# small ones (272), whose calls end after one iteration
@pytest.mark.parametrize("make,small,large", [(_relaxation, (17, 17), (65, 128)), (_projection, (17, 17), (65, 64))])
def test_threads_solve_at_once(make, small, large):
    errors, stop = [], threading.Event()
    solve = make(*large)
    want = solve()
    torch.cuda.synchronize()

    def hammer():
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                short = make(*small, max_it=1)
                while not stop.is_set():
                    try:
                        short()
                    except pg.PdfError as e:
                        if e.status != pg.capi.PDF_ENOTCONV:
                            raise
        except Exception as e:  # reported by the test's own thread
            errors.append(e)

    threads = [threading.Thread(target=hammer) for _ in range(6)]
    for t in threads:
        t.start()
    try:
        same = all(torch.equal(solve(), want) for _ in range(600))
    finally:
        stop.set()
        for t in threads:
            t.join()
    assert not errors
    assert same
