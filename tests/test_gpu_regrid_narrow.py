"""The per-row output onto few output channels: values at the edges of the narrow
form (one and two rows a thread, one column to the last that is narrow and the
first that is not, arrays off the boundaries of its whole loads and stores)
against the 64-bit sums, and its time against a wider output of the same window."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

C_LIGHT = 299792458.0


@pytest.fixture(scope="module")
def V():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_01897_gb300 import build
    build.build()
    from paper_2609_01897_gb300 import vista
    vista.lib()
    return vista


def _off(t, nbytes):
    """The same values in memory that starts nbytes past an allocation's start."""
    k = nbytes // t.element_size()
    return torch.cat([torch.zeros(k, dtype=t.dtype, device=t.device), t.reshape(-1)])[k:].view(t.shape)


CASES = [("c64", 1, 3, 16, 1), ("c64", 4, 1, 16, 1), ("c64", 2, 129, 33, 63), ("c64", 2, 130, 33, 64), ("c64", 4, 257, 40, 31),
         ("c64", 4, 256, 40, 32), ("c64", 2, 90, 40, 29), ("c64", 2, 90, 40, 28), ("c64", 4, 77, 500, 16), ("f16", 1, 3000, 900, 130), ("c64", 1, 700, 64, 127), ("c64", 1, 33333, 20, 7), ("f16", 4, 50001, 12, 4),
         ("bf16", 2, 28573, 9, 7), ("c128", 4, 66667, 8, 3), ("c128", 1, 300, 17, 5), ("f16", 1, 100001, 8, 2)]


# off: bytes of (vis, flags, out_vis, out_wsum) past a 16-byte boundary ("elem": one stored value, one flag)
@pytest.mark.parametrize("off", [None, "elem"])
@pytest.mark.parametrize("vt,npol,nrow,nchan,nrest", CASES)
def test_values(V, vt, npol, nrow, nchan, nrest, off):
    g = torch.Generator(device="cuda")
    g.manual_seed(nrow)
    z, l, m = 0.3, 2e-4, -1e-4
    f = 100e9 + 1e7 * np.arange(nchan)
    uvw = (torch.rand((nrow, 3), generator=g, device="cuda", dtype=torch.float64) - 0.5) * 600.0
    vis = torch.complex(torch.randn((nrow, nchan, npol), generator=g, device="cuda"),
                        torch.randn((nrow, nchan, npol), generator=g, device="cuda"))
    stored, scale = vis, 1.0
    if vt == "c128":
        stored = vis.to(torch.complex128)
    elif vt != "c64":
        scale = 0.25
        stored = (torch.view_as_real(vis) / scale).to(torch.float16 if vt == "f16" else torch.bfloat16)
        vis = torch.view_as_complex((stored.float() * scale).contiguous())
    flags = (torch.rand((nrow, nchan, npol), generator=g, device="cuda") < 0.2).to(torch.uint8)
    out = (torch.full((nrow, nrest, npol, 2), 7.0, device="cuda"), torch.full((nrow, nrest, npol), 7.0, device="cuda"))
    if off:
        stored = _off(stored, {"c64": 8, "c128": 16, "f16": 4, "bf16": 4}[vt])
        flags = _off(flags, 1)
        out = (_off(out[0], 4), _off(out[1], 4))
    rdf = 1.07e7 * (1 + z) * max(0.5, nchan / nrest)
    rf0 = 100e9 * (1 + z) - 0.31 * rdf
    st = V.Stack(4, 4, nrest, 4, 100.0, 100.0, rest_f0=rf0, rest_df=rdf)
    try:
        ov, ow, _ = st.regrid_rows(uvw, f, stored.contiguous(), flags, z=z, l=l, m=m, vis_scale=scale, out=out)
    finally:
        st.close()
    j0, nb, w = V.plan_channels(f, z, rf0, rdf, nrest)
    tau = uvw[:, 0] * l + uvw[:, 1] * m + uvw[:, 2] * (np.sqrt(1.0 - l * l - m * m) - 1.0)
    num = torch.zeros((nrow, nrest, npol), dtype=torch.complex128, device="cuda")
    den = torch.zeros((nrow, nrest, npol), dtype=torch.float64, device="cuda")
    size = torch.zeros_like(den)
    ok = (flags == 0).double()
    for k in range(nchan):
        ph = torch.exp(2j * np.pi * (tau * (f[k] / C_LIGHT)))
        x = vis[:, k].to(torch.complex128) * ph[:, None] * ok[:, k]
        for b in range(nb[k]):
            wk = float(np.float32(w[k, b]))
            num[:, j0[k] + b] += wk * x
            den[:, j0[k] + b] += wk * ok[:, k]
            size[:, j0[k] + b] += wk * x.abs()
    got, gw = torch.view_as_complex(ov.clone()).to(torch.complex128), ow.double()
    has = den > 0
    assert bool(has.any()) and bool(((gw - den).abs() <= 1e-6 * den).all())
    assert bool((got[~has] == 0).all())
    # phasors within 5e-7 rad, then a few roundings of 6e-8
    err = (got[has] - num[has] / den[has]).abs()
    assert bool((err <= 1e-6 * (size[has] / den[has]) + 1e-12).all()), float((err / (size[has] / den[has])).max())


def test_one_channel_is_not_slower_than_many(V):
    """Onto one output channel the window is read once and next to nothing is written: no
    more than four times the time of 64 output channels (it was fifteen)."""
    nrow, nchan = 200000, 64
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    uvw = (torch.rand((nrow, 3), generator=g, device="cuda", dtype=torch.float64) - 0.5) * 600.0
    vis = torch.complex(torch.randn((nrow, nchan, 1), generator=g, device="cuda"), torch.randn((nrow, nchan, 1), generator=g, device="cuda"))
    f = 100e9 + 1e7 * np.arange(nchan)
    times = {}
    for nrest in (1, 64):
        st = V.Stack(4, 4, nrest, 1, 100.0, 100.0, rest_f0=100e9 - 5e6, rest_df=64e7 / nrest)
        out = (torch.empty((nrow, nrest, 1, 2), device="cuda"), torch.empty((nrow, nrest, 1), device="cuda"))
        t = []
        for _ in range(9):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            st.regrid_rows(uvw, f, vis, z=0.0, l=1e-4, out=out)
            b.record()
            b.synchronize()
            t.append(a.elapsed_time(b))
        times[nrest] = sorted(t)[4]
        st.close()
    assert times[1] < 4 * times[64], times
