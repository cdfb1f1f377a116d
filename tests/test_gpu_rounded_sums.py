"""vista_read_cube() and vista_read_cube_sparse() of the mixed cube give the FP64
sum of each entry's FP32 partial and FP64 master, rounded to FP32: bit for bit
the values of vista_read_cube_f64() rounded, also where partial and master
cancel to a small part of either (the FP32 sums of the last run against masters
that hold the runs before, folded)."""
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


# what the second run adds: other data, or the first run's values negated but for a part in 2^10 or 2^18
@pytest.mark.parametrize("left", [None, 2.0 ** -10, 2.0 ** -18])
@pytest.mark.parametrize("npol", [1, 2, 4])
def test_readback_is_the_rounded_fp64_sum(V, npol, left):
    nu, nchan, nrow = 32, 32, 4096
    rng = np.random.default_rng(9)
    uvw = torch.as_tensor(rng.uniform(-30.0, 30.0, (nrow, 3)), device="cuda")
    f = 100e9 + 1e7 * np.arange(nchan)
    g = torch.Generator(device="cuda")
    g.manual_seed(4)
    shape = (nrow, nchan, npol)
    vis = torch.complex(torch.randn(shape, generator=g, device="cuda"), torch.randn(shape, generator=g, device="cuda"))
    wts = torch.rand((nrow, npol), generator=g, device="cuda") + 0.5
    du = 2 * 31.0 * f[-1] / H.C_LIGHT / nu
    st = V.Stack(nu, nu, nchan, npol, du, du, rest_f0=100e9 - 4e6, rest_df=1e7)
    # flagged rows: nothing is stacked, but the visibilities read bring on the fold
    nf = 64 * nu * nu
    fl = (torch.zeros((nf, 3), dtype=torch.float64, device="cuda"), f,
          torch.zeros((nf, nchan, npol), dtype=torch.complex64, device="cuda"), torch.ones((nf, npol), device="cuda"),
          torch.ones((nf, nchan, npol), dtype=torch.uint8, device="cuda"))
    # masters of many significant bits: runs of decreasing size, folded one by one
    sizes = (1.0, 0.77 * 2.0 ** -9, 0.61 * 2.0 ** -17, 0.53 * 2.0 ** -25)
    try:
        for a in sizes:
            st.add_source(uvw, f, vis * a, wts, z=0.0, l=1e-4)
            st.run()
            st.add_source(*fl, z=0.0)
            st.run()
        if left is None:
            st.add_source(uvw.flip(0).contiguous(), f, vis * 0.013, wts, z=0.0, l=1e-4)
        else:
            part = sum(sizes) * (1.0 + left * (2 * torch.rand(shape, generator=g, device="cuda", dtype=torch.float64) - 1))
            st.add_source(uvw, f, (-vis.to(torch.complex128) * part).to(torch.complex64), wts, z=0.0, l=1e-4)
        st.run()
        a = {k: x.cpu().numpy() for k, x in st.read_cube().items()}
        d = {k: x.cpu().numpy() for k, x in st.read_cube(f64=True).items()}
        sp = {k: x.cpu().numpy() for k, x in st.read_cube_sparse().items()}
    finally:
        st.close()
    assert (a["count"] > 0).sum() > 10000
    if left is not None:
        sc = np.sqrt(d["sum_w"] * d["sum_wvv"])[..., None]
        assert np.median(np.abs(d["sum_wv"])[a["count"] > 0] / np.broadcast_to(sc, d["sum_wv"].shape)[a["count"] > 0]) < 4 * left
    for k in ("sum_wv", "sum_w", "sum_wvv"):
        np.testing.assert_array_equal(a[k], d[k].astype(np.float32), err_msg=k)
        np.testing.assert_array_equal(sp[k], a[k].reshape((-1, 2) if k == "sum_wv" else -1)[sp["index"]], err_msg=k)
