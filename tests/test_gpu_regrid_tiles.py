"""The per-row output at the edges of its tiles and tables, against the oracle
and the planner: row counts around a tile of 4 or 8 rows, blocks of columns
partly filled, rest channels narrower and much wider than an input channel,
irregular and descending axes, every storage type."""
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


def _axis(nchan, kind):
    rng = np.random.default_rng(nchan)
    step = np.full(nchan, 2e6) if kind != "irregular" else rng.uniform(0.6e6, 2e6, nchan)
    f = 100e9 + np.cumsum(step)
    return f[::-1].copy() if kind == "descending" else f


# rows: one, around the tiles, and enough of them for the eight-row tiles
@pytest.mark.parametrize("nrow,nchan,npol", [(1, 2, 1), (3, 33, 2), (4, 64, 4), (5, 65, 1), (9, 130, 4),
                                             (5001, 96, 2), (4870, 61, 4)])
@pytest.mark.parametrize("coarse,axis", [(0.35, "even"), (1.0, "descending"), (1.0, "irregular"), (3.7, "irregular"),
                                         (41.0, "even")])
@pytest.mark.parametrize("storage", ["c64", "c128", "f16", "bf16"])
def test_regrid_tiles(V, nrow, nchan, npol, coarse, axis, storage):
    f = _axis(nchan, axis)
    z, l, m = 0.8, 3e-5, -2e-5
    g = torch.Generator(device="cuda")
    g.manual_seed(nrow)
    shape = (nrow, nchan, npol)
    vis = torch.complex(torch.randn(shape, generator=g, device="cuda"), torch.randn(shape, generator=g, device="cuda"))
    uvw = (torch.rand((nrow, 3), generator=g, device="cuda", dtype=torch.float64) - 0.5) * 2000.0
    flags = (torch.rand(shape, generator=g, device="cuda") < 0.1).to(torch.uint8) if npol != 2 else None
    data, scale = vis, 1.0
    if storage == "c128":
        data = vis.to(torch.complex128)
    elif storage != "c64":
        data, scale, _ = H.quantise(vis, storage)
    exact = (torch.view_as_complex(data.double() * scale) if data.dim() == 4 else data.to(torch.complex128)).cpu().numpy()
    rest_df = 2e6 * (1 + z) * coarse
    nrest = int(1.2 * nchan / coarse) + 2
    f0 = f.min() * (1 + z) - 0.7 * rest_df
    for mode in (V.BIN_OVERLAP, V.BIN_NEAREST):
        st = V.Stack(4, 4, nrest, 4, 1.0, 1.0, rest_f0=f0, rest_df=rest_df, bin_mode=mode)
        try:
            got, wsum, uv = st.regrid_rows(uvw, f, data, flags, l=l, m=m, z=z, vis_scale=scale, with_uvw=True)
        finally:
            st.close()
        src = H.O.Source(uvw.cpu().numpy(), f, exact, np.ones((nrow, npol), dtype=np.float32),
                         None if flags is None else flags.cpu().numpy(), l, m, z)
        o_vis, o_w = H.O.regrid_rows(src, f0, rest_df, nrest, mode)
        np.testing.assert_allclose(wsum.cpu().numpy(), o_w, rtol=1e-6, atol=1e-7)
        # as in test_gpu_regrid: a phasor within 5e-7 rad, FP32 sums of a few terms
        err = np.abs(got.cpu().numpy() - o_vis)
        assert (err <= 2e-6 * (np.abs(o_vis) + np.abs(exact).max())).all(), err.max()
        np.testing.assert_array_equal(uv.cpu().numpy(), uvw.cpu().numpy() * (1.0 / (1.0 + z)))
        if flags is None:
            # the device's bins and weights are the planner's: the sums agree to the last bit
            j0, nb, w = V.plan_channels(f, z, f0, rest_df, nrest, mode)
            want = np.zeros(nrest, dtype=np.float32)
            for k in range(nchan):
                for b in range(nb[k]):
                    want[j0[k] + b] += np.float32(w[k, b])
            np.testing.assert_array_equal(wsum.cpu().numpy(), np.broadcast_to(want[None, :, None], wsum.shape))


def test_refused_as_by_the_planner(V):
    """A channel over more than four rest bins is refused; one of just over
    three bins' width is taken."""
    uvw = torch.zeros((2, 3), dtype=torch.float64, device="cuda")
    vis = torch.ones((2, 8, 1), dtype=torch.complex64, device="cuda")
    f = 100e9 + 1e6 * np.arange(8)
    for bins, ok in ((5.5, False), (3.05, True)):
        st = V.Stack(4, 4, 64, 1, 1.0, 1.0, rest_f0=100e9 - 1e6 + 0.01 * 1e6 / bins, rest_df=1e6 / bins)
        try:
            refused = False
            try:
                V.plan_channels(f, 0.0, 100e9 - 1e6 + 0.01 * 1e6 / bins, 1e6 / bins, 64)
            except V.VistaError as e:
                refused = e.code == V.E_RANGE
            assert refused == (not ok)
            if ok:
                st.regrid_rows(uvw, f, vis, z=0.0)
            else:
                with pytest.raises(V.VistaError) as ei:
                    st.regrid_rows(uvw, f, vis, z=0.0)
                assert ei.value.code == V.E_RANGE
        finally:
            st.close()
