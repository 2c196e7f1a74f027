"""First calls on a stream that does not wait for the legacy one, while that one
is kept busy: meshes, hierarchies and work space are in place before the
caller's stream uses them, so the results are those of the default stream, bit
for bit."""
import threading

import pytest

import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1006_0720_gb300 as pg  # noqa: E402


class _BusyDefaultStream:
    """Another thread queues short waits on the default stream."""

    def __enter__(self):
        self.stop = threading.Event()
        self.thread = threading.Thread(target=self._run)
        self.thread.start()

    def _run(self):
        stream = torch.cuda.default_stream()
        with torch.cuda.stream(stream):
            while not self.stop.is_set():
                for _ in range(2):
                    torch.cuda._sleep(200000)  # about 0.1 ms each
                stream.synchronize()

    def __exit__(self, *a):
        self.stop.set()
        self.thread.join()


def _solves(m):
    gm = pg.Mesh(m)
    gp = pg.Particles(gm, 3, ppe=30, u_sigma=0.1)
    pg.pdf_estimate_stats(gp, gm)
    wp = torch.zeros((9, gm.n_nodes), dtype=torch.float64, device="cuda")
    it = pg.pdf_relax_solve_particles(gp, gm, pg.model_params(closure="glm"), wp, rtol=1e-12, max_it=500)
    p = pg.model_params(closure="glm", pressure="projection")
    jt = pg.pdf_pressure_project(gp, gm, p, rtol=1e-10, max_it=500)
    pg.pdf_redistribute(gp, gm, 4, 1, 0)
    return [wp, pg.pdf_pressure_field(gp, gm)] + list(gp.get_state().values()), it, jt


# unknowns of both solves: the cluster forms, and the kernels per sweep
@pytest.mark.parametrize("nx,ny", [(20, 40), (65, 129)])
def test_first_solves_on_a_side_stream(nx, ny):
    m = inputs.channel_mesh(nx, ny, seed=4)
    want, it, jt = _solves(m)
    side = torch.cuda.Stream()
    for _ in range(3):
        with _BusyDefaultStream():
            with torch.cuda.stream(side):
                got, it2, jt2 = _solves(m)
                side.synchronize()
        assert it2 == it and jt2 == jt
        for a, b in zip(want, got):
            assert torch.equal(a, b)


def test_network_parameters_on_a_side_stream():
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    X, Y = torch.randn((256, 11), generator=g, device="cuda"), torch.randn((256, 9), generator=g, device="cuda")
    net = pg.Mlp(1)
    net.fit_norm(X, Y)
    flat, _ = net.params()
    torch.cuda.synchronize()
    want = net.grad(X, Y)
    side = torch.cuda.Stream()
    with _BusyDefaultStream():
        with torch.cuda.stream(side):
            for _ in range(5):
                net.set_params(flat)
                got = net.grad(X, Y)
                side.synchronize()
                assert got[0] == want[0] and (got[1] == want[1]).all()
