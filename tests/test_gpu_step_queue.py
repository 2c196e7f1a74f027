"""The FP32-state step with its walks collected per warp (states of at least
eight rounds of the grid) against the same step in chunks too small for that
(pdf_step_host): the same state and event counts, bit for bit, for whole and
ragged last rounds, with walls, periodic and open boundaries, re-entry and the
concentrated source."""
import numpy as np
import pytest

import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1006_0720_gb300 as pg  # noqa: E402
from paper_1006_0720_gb300 import capi  # noqa: E402


def _round():
    """Particles of one round of the step's grid: 16 blocks of 256 per SM."""
    return 16 * 256 * torch.cuda.get_device_properties(0).multi_processor_count


# (mesh, particles beyond eight rounds): the last size without the queue, a
# whole number of rounds, one particle more, a ragged warp
@pytest.mark.parametrize("mesh,extra", [("channel", -1), ("channel", 0), ("channel", 1), ("obstacles", 12345)])
def test_collected_walks_match_direct_walks(mesh, extra):
    if mesh == "channel":
        m = inputs.channel_mesh(20, 40, seed=1)
        p = pg.model_params(closure="slm")
    else:
        m = inputs.obstacle_mesh(h_min=0.05, ratio=8.0, growth=1.2)
        p = pg.model_params(closure="slm", Pi=2e-2, tm_mode="source", src_x=2.0, src_y=0.5, src_r=0.3)
    gm = pg.Mesh(m)
    n = 8 * _round() + extra
    counts = np.full(gm.n_tri, n // gm.n_tri, dtype=np.int32)
    counts[: n - int(counts.sum())] += 1
    a, b = (pg.Particles(gm, 5, count=counts, u_sigma=0.5, precision=capi.PDF_FP32_STATE) for _ in range(2))
    assert a.n == n
    for q in (a, b):
        pg.pdf_estimate_stats(q, gm)
    host = {k: v.cpu().pin_memory() for k, v in b.get_state().items()}
    for s in range(2):
        a.set_state({k: v.cuda() for k, v in host.items()})  # (positions in the caller's FP64 form on both sides)
        ia = pg.pdf_step(a, gm, p, step=s, info=True)
        ib = pg.pdf_step_host(b, gm, p, host, step=s, info=True)
        assert ia == ib, s
        assert ia["walk_steps"] > n // 100
        got = a.get_state()
        for k, v in host.items():
            assert torch.equal(got[k].cpu(), v), (s, k)
        for q in (a, b):
            pg.pdf_estimate_stats(q, gm)
