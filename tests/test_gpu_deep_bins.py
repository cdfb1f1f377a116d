"""Depth on lattices where a rest bin may be no channel's first: the checkpoints
that keep an entry's FP32 sum short have to reach every bin a run is spread over.
Constant weights and visibilities, every row a run of its own (one row an item):
an entry that is never checkpointed then adds one constant tens of thousands of
times in FP32, and loses up to half a unit in the last place of the total each
time (1e-4 of sum_w at this depth).  With checkpoints the partial sum holds about
g = 8 x pols x bins additions (at most 8 x 4 x 3 = 96 here), each off by at most
half a unit in its last place, 2^-24 g = 5.7e-6 of the sum if every rounding went
the same way: inside the 1e-5 of the mixed path."""
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


# rest bin width in channels: two aligned bins a channel (all odd bins are only
# second bins; sizes that are exact in FP64, so no channel touches a third), two
# or three, three or four, and equal widths a third of a bin apart (the last bin)
@pytest.mark.parametrize("width,offset", [(0.5, 0.0), (0.7, 0.13), (0.4, 0.05), (1.0, 0.375)])
@pytest.mark.parametrize("npol", [1, 2, 4])
def test_every_bin_is_checkpointed(V, npol, width, offset):
    nrow, nchan, df, f0 = 60000, 8, float(2 ** 21), float(2 ** 36)
    rng = np.random.default_rng(5)
    uvw = torch.as_tensor(rng.uniform(-3.0, 3.0, (nrow, 3)), device="cuda")
    f = f0 + df * np.arange(nchan)
    vis = torch.full((nrow, nchan, npol), complex(1.13, 0.37), dtype=torch.complex64, device="cuda")
    wts = torch.full((nrow, npol), 0.7345, device="cuda")
    nrest = int(np.ceil(nchan / width)) + 2
    du = 4.0 * f[-1] / H.C_LIGHT
    out = []
    for prec in (V.PREC_MIXED, V.PREC_FP64):
        st = V.Stack(2, 2, nrest, npol, du, du, rest_f0=f0 - 0.5 * df - offset * df, rest_df=width * df, precision=prec)
        try:
            st.set_tuning(rows_per_item=1)
            st.add_source(uvw, f, vis, wts, z=0.0, l=1e-5, m=2e-5)
            st.run()
            out.append({k: v.cpu().numpy().astype(np.float64) for k, v in st.read_cube(f64=True).items()})
        finally:
            st.close()
    m, r = out
    assert np.array_equal(m["count"], r["count"]) and r["count"].max() >= nrow // 5
    deep = r["count"] > 1000
    assert (deep.any(axis=(0, 1, 3))).sum() >= nchan / width - 1
    scale = {"sum_w": r["sum_w"], "sum_wvv": r["sum_wvv"], "sum_wv": np.sqrt(r["sum_w"] * r["sum_wvv"])[..., None]}
    for k, sc in scale.items():
        err = np.abs(m[k] - r[k])
        assert (err <= H.TOL_MIXED * sc).all(), (k, float((err / np.maximum(sc, 1e-30)).max()))
