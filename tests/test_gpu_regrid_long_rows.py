"""The per-row output of rows longer than 4 GiB (their offsets do not fit 32
bits): onto more than 128 columns, each row's last channels, which lie past that
offset, against the 64-bit sums."""
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


def test_rows_past_four_gib(V):
    npol, nrow, nrest, df, f0 = 4, 2, 40, 64.0, 64e9
    nchan = 2 ** 32 // (16 * npol) + 1000
    f = f0 + df * np.arange(nchan)
    k0 = nchan - nrest   # the output channels are the last 40 channels
    g = torch.Generator(device="cuda")
    g.manual_seed(6)
    uvw = (torch.rand((nrow, 3), generator=g, device="cuda", dtype=torch.float64) - 0.5) * 600.0
    vis = torch.zeros((nrow, nchan, npol), dtype=torch.complex128, device="cuda")
    tail = torch.complex(torch.randn((nrow, nrest, npol), generator=g, device="cuda"),
                         torch.randn((nrow, nrest, npol), generator=g, device="cuda"))
    vis[:, k0:] = tail
    l, m = 2e-4, -1e-4
    st = V.Stack(4, 4, nrest, npol, 100.0, 100.0, rest_f0=f[k0] - 0.5 * df, rest_df=df)
    try:
        out, wsum, _ = st.regrid_rows(uvw, f, vis, z=0.0, l=l, m=m)
    finally:
        st.close()
    tau = uvw[:, 0] * l + uvw[:, 1] * m + uvw[:, 2] * (np.sqrt(1.0 - l * l - m * m) - 1.0)
    want = tail.to(torch.complex128) * torch.exp(2j * np.pi * (tau[:, None] * torch.as_tensor(f[k0:] / C_LIGHT, device="cuda")))[..., None]
    # (channel and lattice edges are multiples of 32 Hz: exact, a channel reaches one bin with weight 1)
    assert bool((wsum == 1.0).all())
    # the phasors within 5e-7 rad, rounding 6e-8 a few times
    assert bool(((out.to(torch.complex128) - want).abs() <= 1e-6 * tail.abs()).all())
