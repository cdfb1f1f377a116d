"""Readback of some of the arrays: the same values as the whole readback, and
not the time of it.  The counts alone are 8 bytes an entry moved where all arrays of
a touched FP64 cube are 60, so they may take no more than half as long."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

from tests import gpu_helpers as H  # noqa: E402

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


def _stacked(V, prec, nu, nrest, npol, nrow, runs):
    rng = np.random.default_rng(3)
    f = 100e9 + 1e7 * np.arange(nrest)
    du = 2 * 31.0 * f[-1] / H.C_LIGHT / nu
    st = V.Stack(nu, nu, nrest, npol, du, du, rest_f0=100e9 - 4e6, rest_df=1e7, precision=prec)
    g = torch.Generator(device="cuda")
    g.manual_seed(2)
    for _ in range(runs):
        uvw = torch.as_tensor(rng.uniform(-30.0, 30.0, (nrow, 3)), device="cuda")
        shape = (nrow, nrest, npol)
        vis = torch.complex(torch.randn(shape, generator=g, device="cuda"), torch.randn(shape, generator=g, device="cuda"))
        st.add_source(uvw, f, vis, torch.rand((nrow, npol), generator=g, device="cuda") + 0.5, z=0.0, l=1e-4)
        st.run()
    return st


# one tile of 1024 entries not filled, just past one, and several rounds of the grid's 152 x 16 tiles
@pytest.mark.parametrize("nu,nrest,npol,nrow,runs", [(2, 3, 1, 50, 1), (8, 17, 1, 3000, 30), (160, 32, 4, 4000, 2)])
@pytest.mark.parametrize("fp64", [False, True])
@pytest.mark.parametrize("f64", [False, True])
def test_parts_equal_the_whole(V, fp64, f64, nu, nrest, npol, nrow, runs):
    st = _stacked(V, V.PREC_FP64 if fp64 else V.PREC_MIXED, nu, nrest, npol, nrow, runs)
    try:
        whole = st.read_cube(f64=f64)
        assert int((whole["count"] > 0).sum()) > 0
        for which in [(k,) for k in KEYS] + [("sum_wv", "count"), ("sum_w", "sum_wvv")]:
            part = st.read_cube(f64=f64, which=which)
            assert set(part) == set(which)
            for k in which:
                assert torch.equal(part[k], whole[k]), (which, k)
    finally:
        st.close()


@pytest.mark.parametrize("fp64", [False, True])
def test_sparse_parts_equal_the_whole(V, fp64):
    import ctypes as C
    st = _stacked(V, V.PREC_FP64 if fp64 else V.PREC_MIXED, 20, 23, 2, 2000, 3)
    try:
        whole = st.read_cube_sparse(device=True)
        n, got = C.c_int64(0), int(whole["index"].shape[0])
        assert got > 1000
        for which in ((), ("count",), ("sum_w",), ("sum_wvv", "count"), ("sum_wv",)):
            part = {k: torch.full_like(x, 7) for k, x in whole.items()}
            ptr = {k: (x.data_ptr() if k == "index" or k in which else None) for k, x in part.items()}
            rc = V.lib().vista_read_cube_sparse(st.h, got, ptr["index"], ptr["sum_wv"], ptr["sum_w"], ptr["sum_wvv"],
                                                ptr["count"], C.byref(n), 1)
            assert rc == 0 and n.value == got
            for k, x in part.items():
                assert torch.equal(x, whole[k] if ptr[k] else torch.full_like(x, 7)), (which, k)
    finally:
        st.close()


def test_counts_alone_do_not_read_the_sums(V):
    st = _stacked(V, V.PREC_FP64, 256, 64, 4, 40000, 1)
    try:
        times = {}
        for which in (KEYS, ("count",)):
            out = st.read_cube(which=which)
            t = []
            for _ in range(9):
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record()
                st.read_cube(which=which, out=out)
                b.record()
                b.synchronize()
                t.append(a.elapsed_time(b))
            times[which] = sorted(t)[4]
        assert times[("count",)] < 0.5 * times[KEYS], times
    finally:
        st.close()
