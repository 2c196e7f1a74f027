"""A velocity component that is not finite: the particle is counted as lost and
keeps its place, the call says so, and every other particle moves as it does
without it."""
import numpy as np
import pytest

import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1006_0720_gb300 as pg  # noqa: E402
from paper_1006_0720_gb300 import capi  # noqa: E402


@pytest.mark.parametrize("component", ["u", "v"])
@pytest.mark.parametrize("value", [np.nan, np.inf])
@pytest.mark.parametrize("precision", [capi.PDF_FP64, capi.PDF_FP32_STATE])
@pytest.mark.parametrize("host", [False, True])
def test_particle_with_one_component_not_finite_is_lost(component, value, precision, host):
    gm = pg.Mesh(inputs.channel_mesh(12, 16, seed=1))
    p = pg.model_params(closure="glm")
    ends = []
    for spoil in (False, True):
        gp = pg.Particles(gm, 5, ppe=20, u_sigma=0.1, precision=precision)
        pg.pdf_estimate_stats(gp, gm)
        st = gp.get_state()
        bad = gp.n // 2  # away from the walls
        assert abs(float(st["y"][bad])) < 0.5
        if spoil:
            st[component][bad] = value
        before = {k: v.clone() for k, v in st.items()}
        if host:
            arrays = {k: v.cpu().pin_memory() for k, v in st.items()}
            step = lambda: pg.pdf_step_host(gp, gm, p, arrays, step=0, info=True)  # noqa: E731
        else:
            gp.set_state(st)
            step = lambda: pg.pdf_step(gp, gm, p, step=0, info=True)  # noqa: E731
        info = step()
        assert info["lost"] == (1 if spoil else 0)
        assert (info.get("status") == "lost") == spoil  # (the call's own status: PDF_ELOST)
        after = {k: v.cuda() for k, v in (arrays if host else gp.get_state()).items()}
        if spoil:
            for k in ("x", "y", "elem"):
                assert after[k][bad] == before[k][bad], k
        ends.append(after)
    for k in ends[0]:
        keep = torch.ones(gp.n, dtype=torch.bool, device="cuda")
        keep[bad] = False
        assert torch.equal(ends[0][k][keep], ends[1][k][keep]), k
