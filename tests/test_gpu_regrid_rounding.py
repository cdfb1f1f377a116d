"""Rounding of the per-row output: each contribution w (V e^{i phi}) is formed as a
product of V and the phasor, rounded, and added with its weight in one
fused operation.  The phasors are the library's own (exported), so that what is
left against 64 bits is this arithmetic; its rms must be that of the same FP32
operations restated in NumPy (a few per cent allowed for the choice of which
products the restatement fuses; another rounding a contribution adds 10 to 20 %)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def V():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_01897_gb300 import build
    build.build()
    from paper_2609_01897_gb300 import vista
    vista.lib()
    return vista


def _fma(a, b, c):
    return (a.astype(np.float64) * b.astype(np.float64) + c.astype(np.float64)).astype(np.float32)


@pytest.mark.parametrize("npol", [1, 2, 4])
@pytest.mark.parametrize("width,offset", [(0.61, 0.27), (0.93, 0.31)])
def test_rms_of_the_sums(V, npol, width, offset):
    nrow, nchan, df, f0 = 3000, 48, 1e7, 100e9
    g = torch.Generator(device="cuda")
    g.manual_seed(11)
    uvw = (torch.rand((nrow, 3), generator=g, device="cuda", dtype=torch.float64) - 0.5) * 400.0
    f = f0 + df * np.arange(nchan)
    vis = torch.complex(torch.randn((nrow, nchan, npol), generator=g, device="cuda"),
                        torch.randn((nrow, nchan, npol), generator=g, device="cuda"))
    wts = torch.ones((nrow, npol), device="cuda")
    nrest = int(nchan / width) - 2
    rf0, rdf = f0 + offset * df, width * df
    st = V.Stack(64, 64, nrest, 4, 5e3, 5e3, rest_f0=rf0, rest_df=rdf)
    try:
        st.add_source(uvw, f, vis, wts, z=0.0, l=3e-4, m=-2e-4)
        st.run()
        ph = torch.view_as_complex(st.debug_phasors(0, nrow, nchan)).cpu().numpy()
        out, wsum, _ = st.regrid_rows(uvw, f, vis, z=0.0, l=3e-4, m=-2e-4)
        out, wsum = out.cpu().numpy(), wsum.cpu().numpy()
    finally:
        st.close()
    j0, nb, w = V.plan_channels(f, 0.0, rf0, rdf, nrest)
    v = vis.cpu().numpy()
    shape = (nrow, nrest, npol)
    exact, size, sw64 = np.zeros(shape, np.complex128), np.zeros(shape), np.zeros((1, nrest, 1))
    sr, si, sw = np.zeros(shape, np.float32), np.zeros(shape, np.float32), np.zeros((1, nrest, 1), np.float32)
    c, s = ph.real.astype(np.float32), ph.imag.astype(np.float32)
    assert np.array_equal(c.astype(np.float64), ph.real)
    for k in range(nchan):
        for b in range(nb[k]):
            j, wk = j0[k] + b, np.float32(w[k, b])
            x = np.float64(wk) * v[:, k].astype(np.complex128) * ph[:, k, None]
            exact[:, j] += x
            size[:, j] += np.abs(x)
            sw64[:, j] += np.float64(wk)
            ck, sk = c[:, k, None], s[:, k, None]
            re, im = _fma(v[:, k].real, ck, -(v[:, k].imag * sk)), _fma(v[:, k].real, sk, v[:, k].imag * ck)
            sr[:, j], si[:, j] = _fma(np.full_like(re, wk), re, sr[:, j]), _fma(np.full_like(im, wk), im, si[:, j])
            sw[:, j] += wk
    ok = sw64[0, :, 0] > 0
    assert ok.sum() > 30 and np.array_equal(wsum[:, ok], np.broadcast_to(sw, shape)[:, ok])

    def rms(o):
        e = np.abs(o[:, ok] - exact[:, ok] / sw64[:, ok]) / (size[:, ok] / sw64[:, ok])
        return float(np.sqrt((e ** 2).mean()))

    want = np.zeros(shape, np.complex128)
    want[:, ok] = sr[:, ok] / sw[:, ok] + 1j * (si[:, ok] / sw[:, ok]).astype(np.float64)
    assert rms(out) <= 1.03 * rms(want), (rms(out), rms(want))
