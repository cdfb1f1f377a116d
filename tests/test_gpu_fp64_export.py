"""vista_debug_phasors() and vista_debug_cells() of the FP64 form give what its
stacking kernel uses, bit for bit: unit visibilities of unit weight, each alone in
its cube entry, so that the entry's sum is the phasor itself."""
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


@pytest.mark.parametrize("npol", [1, 2, 4])
@pytest.mark.parametrize("axis", ["linear", "descending", "irregular"])
@pytest.mark.parametrize("fold", [False, True])
def test_export_is_what_the_kernel_uses(V, npol, axis, fold):
    nrow, nchan, nu = 40, 101, 256
    rng = np.random.default_rng(8)
    f = 100e9 + 2e6 * np.arange(nchan)
    if axis == "descending":
        f = f[::-1].copy()
    elif axis == "irregular":
        f = f + rng.uniform(-5e5, 5e5, nchan)
    # rows more than two cells apart along v (of 600 m / 256), either sign; distinct |v| for the fold
    v = (np.arange(nrow) + 0.5) * 7.1 * np.where(rng.random(nrow) < 0.5, -1.0, 1.0)
    uvw = np.stack([rng.uniform(-290.0, 290.0, nrow), v, rng.uniform(-40.0, 40.0, nrow)], 1)
    du = 602.0 * f.max() / H.C_LIGHT / nu
    st = V.Stack(nu, nu, nchan, npol, du, du, rest_f0=100e9 - 1e6, rest_df=2e6, bin_mode=V.BIN_NEAREST,
                 precision=V.PREC_FP64, hermitian_fold=fold)
    vis, wts = torch.ones((nrow, nchan, npol), dtype=torch.complex64, device="cuda"), torch.ones((nrow, npol), device="cuda")
    base = torch.as_tensor(uvw, device="cuda")   # (kept: the exports read the window's arrays)
    try:
        st.add_source(base, f, vis, wts, z=0.0, l=3e-4, m=-2e-4)
        st.run()
        cube = {k: x.cpu().numpy() for k, x in st.read_cube(f64=True).items()}
        ph = st.debug_phasors(0, nrow, nchan).cpu().numpy()
        cells = st.debug_cells(0, nrow, nchan).cpu().numpy()
    finally:
        st.close()
    assert cube["count"].max() == 1 and cube["count"].sum() == nrow * nchan * npol and cells.min() >= 0
    j = np.floor((f - (100e9 - 1e6)) / 2e6).astype(int)
    sign = np.where(fold & (v < 0), -1.0, 1.0)
    for r in range(nrow):
        got = cube["sum_wv"][cells[r, :, 1], cells[r, :, 0], j]
        for p in range(npol):
            np.testing.assert_array_equal(got[:, p, 0], ph[r, :, 0])
            np.testing.assert_array_equal(got[:, p, 1], sign[r] * ph[r, :, 1])
