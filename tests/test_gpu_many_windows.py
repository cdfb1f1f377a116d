"""The row ordering cuts the cube into stripes by the number of windows of a run:
runs of one window, of many small ones and of one again on one handle (32
stripes, one, 32), each also replayed, against the FP64 form."""
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


def _windows(n, nrow, nchan, npol, seed, half):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    f = 100e9 + 1e7 * np.arange(nchan)
    out = []
    for _ in range(n):
        uvw = (torch.rand((nrow, 3), generator=g, device="cuda", dtype=torch.float64) - 0.5) * 2 * half
        vis = torch.complex(torch.randn((nrow, nchan, npol), generator=g, device="cuda"),
                            torch.randn((nrow, nchan, npol), generator=g, device="cuda"))
        out.append((uvw, f, vis, torch.rand((nrow, npol), generator=g, device="cuda") + 0.5))
    return out


@pytest.mark.parametrize("sort_rows", [1, 0])
@pytest.mark.parametrize("many", [39, 100, 1300])
def test_stripes_change_from_run_to_run(V, many, sort_rows):
    nu, nchan, npol, half = 36, 17, 2, 30.0
    sets = [_windows(1, 1500, nchan, npol, 1, half), _windows(many, 7, nchan, npol, 2, half), _windows(1, 900, nchan, npol, 3, half)]
    du = 2 * half * 1.02 * sets[0][0][1][-1] / H.C_LIGHT / nu
    out = []
    for prec in (V.PREC_MIXED, V.PREC_FP64):
        st = V.Stack(nu, nu, nchan, npol, du, du, rest_f0=100e9 - 4e6, rest_df=1e7, precision=prec)
        try:
            st.set_tuning(sort_rows=sort_rows)
            for windows in sets:
                for _ in range(3):   # planned, captured, replayed
                    for u, f, v, w in windows:
                        st.add_source(u, f, v, w, z=0.0, l=1e-4)
                    st.run()
            out.append((st.stats(), {k: x.cpu().numpy().astype(np.float64) for k, x in st.read_cube(f64=True).items()}))
        finally:
            st.close()
    (sm, m), (sr, r) = out
    assert np.array_equal(m["count"], r["count"])
    assert sm["n_stacked"] == sr["n_stacked"] == 3 * (1500 + 7 * many + 900) * nchan * npol
    sc = np.sqrt(r["sum_w"] * r["sum_wvv"])[..., None]
    assert (np.abs(m["sum_wv"] - r["sum_wv"]) <= H.TOL_MIXED * sc).all()
    assert (np.abs(m["sum_w"] - r["sum_w"]) <= H.TOL_MIXED * r["sum_w"]).all()
