"""The grouping by element at the sizes where its plan changes (one or two
passes, digit widths, tile size, tile counts summed by the scatter or
scanned): exact counts and means of particles in no order, and the same bits
from the allocation-free entry point."""
import numpy as np
import pytest

import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1006_0720_gb300 as pg  # noqa: E402


def _state(m, n, seed):
    """n particles at the centroids of randomly chosen elements."""
    rng = np.random.default_rng(seed)
    e = rng.integers(0, len(m["tri"]), n).astype(np.int32)
    c = m["xy"][m["tri"]].mean(axis=1)
    st = dict(x=c[e, 0].copy(), y=c[e, 1].copy(), elem=e)
    for k in ("u", "v", "w", "om", "ps"):
        st[k] = rng.random(n)
    return st


# (nx, ny): 8, 2,048, 2,112 (12 bits), 16,384 (14), 131,072 (17), 264,196 elements
# (19: two digits of ten bits); n: below, at and above one small tile, the last
# size of small tiles, the last with summed counts, and with a scan
@pytest.mark.parametrize("nx,ny,n", [(3, 3, 1), (3, 3, 1024), (33, 33, 1025), (33, 34, 131072), (33, 33, 131073),
                                     (129, 65, 131073), (129, 65, 655360), (33, 33, 655361), (257, 257, 700001),
                                     (3, 66050, 300001)])
def test_grouping_plans(nx, ny, n):
    m = inputs.channel_mesh(nx, ny, seed=1)
    n_tri = len(m["tri"])
    gm = pg.Mesh(m)
    counts = np.zeros(n_tri, dtype=np.int32)
    counts[0] = n
    gp = pg.Particles(gm, 1, count=counts)
    st = _state(m, n, nx + n)
    gp.set_state({k: torch.from_numpy(a).cuda() for k, a in st.items()})
    gp.set_reorder(0)
    outs = [torch.empty((n_tri, 13), dtype=torch.float64, device="cuda") for _ in range(3)]
    pg.pdf_estimate_stats(gp, gm, elem_stats=outs[0])
    N = np.bincount(st["elem"], minlength=n_tri)
    got = outs[0].cpu().numpy()
    assert np.array_equal(got[:, 0], N)
    for q, k in enumerate(("u", "v", "w", "om", "ps")):
        mean = np.bincount(st["elem"], weights=st[k], minlength=n_tri) / np.maximum(N, 1)
        # double-float sums: 2^-46 of the values, which lie in [0, 1)
        assert np.abs(got[:, 1 + q] - mean).max() < 1e-12, k
    if n <= pg.capi.PDF_NOALLOC_MAX_PARTICLES and n_tri <= pg.capi.PDF_NOALLOC_MAX_ELEMENTS:
        pg.pdf_estimate_stats_noalloc(gp, gm, elem_stats=outs[1])
        assert torch.equal(outs[0], outs[1])
    # a copy into element order: the same groups in the same order
    gp.set_reorder(1)
    pg.pdf_estimate_stats(gp, gm, elem_stats=outs[2])
    assert torch.equal(outs[0], outs[2])
    after = gp.get_state()
    for k, a in st.items():
        assert np.allclose(after[k].cpu().numpy(), a, rtol=0, atol=1e-14), k


def test_grouping_with_shared_histograms():
    """Above 8,192 tiles four tiles share a histogram: exact counts, and the same
    statistics to the bit before and after a copy into element order."""
    m = inputs.channel_mesh(129, 65, seed=1)
    n_tri, n = len(m["tri"]), 33600001
    gm = pg.Mesh(m)
    counts = np.zeros(n_tri, dtype=np.int32)
    counts[0] = n
    gp = pg.Particles(gm, 1, count=counts, precision=pg.capi.PDF_FP32_STATE)
    st = _state(m, n, 9)
    gp.set_state({k: torch.from_numpy(a).cuda() for k, a in st.items()})
    a, b = (torch.empty((n_tri, 13), dtype=torch.float64, device="cuda") for _ in range(2))
    gp.set_reorder(0)
    pg.pdf_estimate_stats(gp, gm, elem_stats=a)
    gp.set_reorder(1)
    pg.pdf_estimate_stats(gp, gm, elem_stats=b)
    assert np.array_equal(a[:, 0].cpu().numpy(), np.bincount(st["elem"], minlength=n_tri))
    assert torch.equal(a, b)
    assert np.array_equal(gp.get_state()["elem"].cpu().numpy(), st["elem"])
