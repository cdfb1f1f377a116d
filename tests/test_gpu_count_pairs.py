"""Where runs are not merged (a channel over three or more rest bins, plane maps
that skip a pol), the counts of a pol pair on adjacent planes still take one
reduction: n_reductions of a stack whose runs are known (one row an item, every
visibility a run), and the sums against the FP64 form."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

from tests import gpu_helpers as H  # noqa: E402


@pytest.fixture(scope="module")
def V():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_01897_gb300 import build
    build.build()
    from paper_2609_01897_gb300 import vista
    vista.lib()
    return vista


# map, rest bin width in channels, reductions a run and rest bin: a vector one for
# every mapped pol, a count for every pair on planes (even, next) and for every other mapped pol
@pytest.mark.parametrize("pmap,width,per_bin", [((0, 1), 0.4, 3), ((0, 1, 2, 3), 0.4, 6), ((0, 1, -1, 3), 0.8, 5),
                                                ((2, 3, -1, -1), 0.8, 3), ((1, 2), 0.4, 4), ((-1, -1, 0, 1), 0.4, 3)])
def test_count_reductions(V, pmap, width, per_bin):
    nrow, nchan, npol, planes = 4000, 32, len(pmap), 4 if max(pmap) > 1 or len(pmap) > 2 else 2
    rng = np.random.default_rng(2)
    uvw = torch.as_tensor(rng.uniform(-3.0, 3.0, (nrow, 3)), device="cuda")
    f = 100e9 + 1e7 * np.arange(nchan)
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    shape = (nrow, nchan, npol)
    vis = torch.complex(torch.randn(shape, generator=g, device="cuda"), torch.randn(shape, generator=g, device="cuda"))
    wts = torch.rand((nrow, npol), generator=g, device="cuda") + 0.5
    rf0, rdf, nrest = 100e9 - 5.3e6, 1e7 * width, int(nchan / width) + 2
    du = 4.0 * f[-1] / H.C_LIGHT
    out = []
    for prec in (V.PREC_MIXED, V.PREC_FP64):
        st = V.Stack(4, 4, nrest, planes, du, du, rest_f0=rf0, rest_df=rdf, precision=prec)
        try:
            st.set_tuning(rows_per_item=1)
            st.add_source(uvw, f, vis, wts, z=0.0, l=1e-5, pol_map=list(pmap))
            st.run()
            out.append((st.stats(), {k: x.cpu().numpy().astype(np.float64) for k, x in st.read_cube(f64=True).items()}))
        finally:
            st.close()
    (stats, m), (_, r) = out
    nb = V.plan_channels(f, 0.0, rf0, rdf, nrest)[1]
    assert nb.min() >= 1 and (width != 0.4 or nb.max() >= 3)
    runs = nrow * nchan
    base = nrow * per_bin * int(nb.sum())
    # checkpoints: one drain in eight, five reductions a lane; another count a pair and bin would add runs or more
    assert base <= stats["n_reductions"] <= base + 0.9 * runs, (stats["n_reductions"] - base) / runs
    assert np.array_equal(m["count"], r["count"]) and m["count"].sum() > 0
    sc = np.sqrt(r["sum_w"] * r["sum_wvv"])[..., None]
    assert (np.abs(m["sum_wv"] - r["sum_wv"]) <= H.TOL_MIXED * sc).all()
    assert (np.abs(m["sum_w"] - r["sum_w"]) <= H.TOL_MIXED * r["sum_w"]).all()
