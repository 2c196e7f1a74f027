"""Element statistics on both sides of the line between their overlapped and
their ordinary launch (256 particles per element): exact counts, and means and
variances of particles in no order, in both storage forms."""
import numpy as np
import pytest

import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1006_0720_gb300 as pg  # noqa: E402
from paper_1006_0720_gb300 import capi  # noqa: E402


# 8 elements: 256 particles per element and one more in all; 870 elements likewise, and full
@pytest.mark.parametrize("nx,ny,n", [(3, 3, 2048), (3, 3, 2049), (16, 30, 222720), (16, 30, 222721), (16, 30, 1131000)])
@pytest.mark.parametrize("precision", [capi.PDF_FP64, capi.PDF_FP32_STATE])
def test_statistics_of_full_elements(nx, ny, n, precision):
    m = inputs.channel_mesh(nx, ny, seed=1)
    n_tri = len(m["tri"])
    rng = np.random.default_rng(n)
    e = rng.integers(0, n_tri, n).astype(np.int32)
    c = m["xy"][m["tri"]].mean(axis=1)
    st = dict(x=c[e, 0].copy(), y=c[e, 1].copy(), elem=e)
    for k in ("u", "v", "w", "om", "ps"):
        st[k] = rng.random(n).astype(np.float32).astype(np.float64)  # (the same values in both forms)
    gm = pg.Mesh(m)
    counts = np.zeros(n_tri, dtype=np.int32)
    counts[0] = n
    gp = pg.Particles(gm, 1, count=counts, precision=precision)
    gp.set_state({k: torch.from_numpy(a).cuda() for k, a in st.items()})
    es = torch.empty((n_tri, 13), dtype=torch.float64, device="cuda")
    for every in (0, 1):  # by the sorted slots, and after the copy into element order
        gp.set_reorder(every)
        pg.pdf_estimate_stats(gp, gm, elem_stats=es)
        got = es.cpu().numpy()
        N = np.bincount(e, minlength=n_tri)
        assert np.array_equal(got[:, 0], N)
        D = np.maximum(N, 1)
        for q, k in enumerate(("u", "v", "w", "om", "ps")):
            mean = np.bincount(e, weights=st[k], minlength=n_tri) / D
            # double-float sums of values in [0, 1): 2^-44 of them
            assert np.abs(got[:, 1 + q] - mean).max() < 1e-12, k
            if k in "uvw":
                var = np.bincount(e, weights=(st[k] - mean[e]) ** 2, minlength=n_tri) / D
                assert np.abs(got[:, 6 + q] - var).max() < 1e-11, k
