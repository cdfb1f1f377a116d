"""NaN and infinite visibilities stay visible in what is read back: through the
checkpoints and folds that move FP32 sums into the FP64 master cube, and through
continuum subtraction of the mixed cube (before and after a fold) and of the
FP64 cube.  The rule: a sum that a non-finite visibility has entered is not
finite; a plane of a cell with such a sum among its line-free channels has no
finite fit, so none of its outputs is finite; elsewhere the output is finite
exactly where the sum is."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

from tests import gpu_helpers as H  # noqa: E402

BAD = [complex(float("nan"), 0.0), complex(float("inf"), 0.0), complex(1.0, float("-inf"))]


@pytest.fixture(scope="module")
def V():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_01897_gb300 import build
    build.build()
    from paper_2609_01897_gb300 import vista
    vista.lib()
    return vista


def _window(nrow, nchan, npol, seed, half):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    uvw = (torch.rand((nrow, 3), generator=g, device="cuda", dtype=torch.float64) - 0.5) * 2 * half
    vis = torch.complex(torch.randn((nrow, nchan, npol), generator=g, device="cuda"),
                        torch.randn((nrow, nchan, npol), generator=g, device="cuda"))
    wts = torch.rand((nrow, npol), generator=g, device="cuda") + 0.5
    return uvw, 100e9 + 1e7 * np.arange(nchan), vis, wts


@pytest.mark.parametrize("bad", BAD)
@pytest.mark.parametrize("npol", [1, 2, 4])
def test_through_checkpoints(V, npol, bad):
    """Thousands of drains after the bad value: its entry is checkpointed many times."""
    uvw, f, vis, wts = _window(30000, 8, npol, 3, 30.0)
    vis[11, 3, npol - 1] = bad
    du = 2 * 30.0 * 1.01 * f[-1] / H.C_LIGHT / 2
    got = []
    for prec in (V.PREC_MIXED, V.PREC_FP64):
        st = V.Stack(2, 2, 9, npol, du, du, rest_f0=100e9 - 4e6, rest_df=1e7, precision=prec)
        try:
            st.set_tuning(rows_per_item=1)
            st.add_source(uvw, f, vis, wts, z=0.0, l=1e-4, m=-2e-4)
            st.run()
            got.append([{k: x.cpu().numpy() for k, x in st.read_cube(f64=w).items()} for w in (False, True)])
        finally:
            st.close()
    for g, want in zip(got[0], got[1]):
        for k in ("sum_wv", "sum_w", "sum_wvv"):
            assert np.array_equal(np.isfinite(g[k]), np.isfinite(want[k])), k
        assert not np.isfinite(g["sum_wvv"]).all() and np.isfinite(g["sum_w"]).all()


@pytest.mark.parametrize("bad", BAD)
@pytest.mark.parametrize("planes", [1, 2, 3, 4])
@pytest.mark.parametrize("order", [0, 1, 3])
@pytest.mark.parametrize("in_line", [False, True])
def test_contsub(V, planes, bad, order, in_line):
    npol, nu, nrest = {1: 1, 2: 2, 3: 2, 4: 4}[planes], 4, 33
    uvw, f, vis, wts = _window(300, 33, npol, 7, 30.0)
    vis[1, 16, npol - 1] = bad
    free = np.ones(nrest, dtype=bool)
    if in_line:
        free[15:18] = False   # the bins channel 16 reaches
    du = 2 * 30.0 * 1.01 * f[-1] / H.C_LIGHT / nu
    empty = (torch.zeros((6000, 3), dtype=torch.float64, device="cuda"), f,
             torch.zeros((6000, 33, npol), dtype=torch.complex64, device="cuda"),
             torch.ones((6000, npol), device="cuda"), torch.ones((6000, 33, npol), dtype=torch.uint8, device="cuda"))
    assert 6000 * 31 * npol >= 64 * nu * nu * nrest * planes   # visibilities read, enough for a fold
    out = {}
    for name, prec in (("mixed", V.PREC_MIXED), ("fp64", V.PREC_FP64)):
        st = V.Stack(nu, nu, nrest, planes, du, du, rest_f0=100e9 - 4e6, rest_df=1e7, precision=prec)
        try:
            st.add_source(uvw, f, vis, wts, z=0.0)
            st.run()
            out[name] = (st.read_cube(f64=True), st.contsub(free, order))
            st.add_source(*empty, z=0.0)   # all flagged: only the fold
            st.run()
            out[name + " after a fold"] = (st.read_cube(f64=True), st.contsub(free, order))
        finally:
            st.close()
    base = {k: v.cpu().numpy() for k, v in out["fp64"][0].items()}
    ok = np.isfinite(base["sum_wv"])
    assert not ok.all()
    fit_ok = ok[:, :, free].all(axis=(2, 4), keepdims=True)   # per cell and plane
    bad_plane = ~fit_ok[:, :, 0, :, 0]
    assert bad_plane.any() != in_line
    scale = np.nan_to_num(np.sqrt(base["sum_w"] * base["sum_wvv"]), posinf=0.0).max()
    ref = out["fp64"][1].cpu().numpy()
    for name, (cube, c) in out.items():
        c = c.cpu().numpy()
        # (a component may stay finite where only the other one is not: a value counts as finite if both are)
        both, sums = np.isfinite(c).all(-1), ok.all(-1) & fit_ok[..., 0]
        assert np.array_equal(both, sums), name
        assert np.abs(c[both] - ref[both]).max() <= 1e-4 * scale, name
