"""Readback, zeroing and continuum subtraction skip cube entries whose count
is 0.  Against the general form (every entry read), which a handle takes once
its counts may have wrapped: windows whose visibilities are all flagged raise
the bound on the counts past 2^32 without touching an entry."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

KEYS = ("sum_wv", "sum_w", "sum_wvv", "count")


@pytest.fixture(scope="module")
def V():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_01897_gb300 import build
    build.build()
    from paper_2609_01897_gb300 import vista
    vista.lib()
    return vista


def _window(nrow, nchan, npol, seed, bad=None):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    uvw = (torch.rand((nrow, 3), generator=g, device="cuda", dtype=torch.float64) - 0.5) * 60.0
    vis = torch.complex(torch.randn((nrow, nchan, npol), generator=g, device="cuda"),
                        torch.randn((nrow, nchan, npol), generator=g, device="cuda"))
    if bad is not None:
        vis[1, nchan // 2, 0] = bad
    wts = torch.rand((nrow, npol), generator=g, device="cuda") + 0.5
    f = 100e9 + 1e7 * np.arange(nchan)
    return uvw, f, vis, wts


def _raise_bound(V, st):
    """Queue all-flagged windows (nothing is stacked) until 2^32 is passed:
    16384 rows x 1024 channels in one rest bin, 256 times."""
    nrow, nchan = 16384, 1024
    uvw = torch.zeros((nrow, 3), dtype=torch.float64, device="cuda")
    vis = torch.zeros((nrow, nchan, 1), dtype=torch.complex64, device="cuda")
    wts = torch.ones((nrow, 1), device="cuda")
    flags = torch.ones((nrow, nchan, 1), dtype=torch.uint8, device="cuda")
    f = 100.1e9 + 1.0 * np.arange(nchan)
    for _ in range(257):
        st.add_source(uvw, f, vis, wts, flags, z=0.0)
    st.run()
    st.stats()


# entries: below, at and off a multiple of the kernels' 1024-entry tile; one
# cell of more than one 256-entry group; the per-plane contsub (npol 3)
@pytest.mark.parametrize("nu,nrest,npol", [(2, 1, 1), (16, 4, 1), (10, 37, 2), (6, 131, 4), (8, 21, 3)])
@pytest.mark.parametrize("fp64", [False, True])
@pytest.mark.parametrize("bad", [None, complex(float("nan"), 0.0), complex(float("inf"), 0.0)])
def test_guarded_equals_general(V, nu, nrest, npol, fp64, bad):
    st = V.Stack(nu, nu, nrest, npol, 20000.0 / nu, 20000.0 / nu, rest_f0=100e9 - 5e6, rest_df=max(3.7e8 / nrest, 4e6),
                 precision=V.PREC_FP64 if fp64 else V.PREC_MIXED)
    pin = {1: 1, 2: 2, 3: 2, 4: 4}[npol]
    uvw, f, vis, wts = _window(150, 33, pin, 7, bad)
    lf = np.ones(nrest, dtype=bool)
    try:
        st.add_source(uvw, f, vis, wts, z=0.0)
        st.run()

        def products():
            # (no continuum subtraction of a non-finite sum: raising the bound below also folds the FP32
            # sums, and the subtraction takes a non-finite FP64 master as 0 but a non-finite FP32 sum as it is)
            return [st.read_cube(), st.read_cube(f64=True)] + (
                [{"c1": st.contsub(lf, 1), "c0": st.contsub(lf, 0)}] if bad is None else [])

        got = products()
        off = torch.zeros(2 * nu * nu * nrest * npol + 1, device="cuda")[1:].view(nu, nu, nrest, npol, 2)
        odd = st.read_cube(which=("sum_wv",), out={"sum_wv": off})["sum_wv"]
        assert torch.equal(torch.nan_to_num(odd), torch.nan_to_num(got[0]["sum_wv"]))
        _raise_bound(V, st)
        want = products()
        assert 0 < int((got[0]["count"] > 0).sum())
        for a, b in zip(got, want):
            for k in a:
                np.testing.assert_array_equal(a[k].cpu().numpy(), b[k].cpu().numpy(), err_msg=k)
        # FP32 sums are the FP64 sums rounded (one unit in the last place allowed)
        for k in KEYS[:3]:
            a, d = got[0][k].double().cpu().numpy(), got[1][k].float().double().cpu().numpy()
            with np.errstate(invalid="ignore"):
                assert (np.isclose(a, d, rtol=1.2e-7, atol=0.0, equal_nan=True)).all(), k
        # zeroing, general (bound past 2^32) and then guarded: the same stack again is the same cube
        for _ in range(2):
            st.zero()
            z = st.read_cube()
            assert all(int((z[k] != 0).sum()) == 0 for k in KEYS)
            st.add_source(uvw, f, vis, wts, z=0.0)
            st.run()
            again = st.read_cube()
            assert torch.equal(again["count"], got[0]["count"])
            # the order of the atomics varies: FP32 sums of at most 150 x 33 terms
            np.testing.assert_allclose(again["sum_w"].cpu().numpy(), got[0]["sum_w"].cpu().numpy(), rtol=1e-5)
    finally:
        st.close()
