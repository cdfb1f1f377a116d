"""Runs whose windows need several stacking kernels (pols, stored types, chunk
widths) share one row-ordering pre-pass: device windows at once, host windows
wave by wave, in cell order and in row order, mixed and FP64, replayed."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

from tests import gpu_helpers as H  # noqa: E402

LINE, DF = 230e9, 4e6


@pytest.fixture(scope="module")
def V():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_01897_gb300 import build
    build.build()
    from paper_2609_01897_gb300 import vista
    vista.lib()
    return vista


def _workload(windows):
    """windows: (rows, channels, pols, complex128?)"""
    from paper_2609_01897_gb300 import synth
    rest_df = DF * 1.7
    wl = synth.Workload("classes", 24, 24, 150, 4, 4.0, 4.0, LINE, [], rest_df=rest_df, rest_f0=LINE - 75 * rest_df)
    for k, (n, nchan, npol, wide) in enumerate(windows):
        rng = np.random.default_rng([k, n, nchan])
        z = 0.7
        f = LINE / (1 + z) + DF * (np.arange(nchan) - 0.5 * nchan)
        wl.du = wl.dv = 2 * 330.0 * LINE / (1 + z) / H.C_LIGHT / 24
        uvw = np.concatenate([rng.uniform(-300, 300, (n, 2)), rng.uniform(-30, 30, (n, 1))], 1)
        g = torch.Generator(device="cuda")
        g.manual_seed(100 * k + n)
        shape = (n, nchan, npol)
        vis = torch.complex(torch.randn(shape, generator=g, device="cuda"), torch.randn(shape, generator=g, device="cuda"))
        wts = torch.rand((n, npol), generator=g, device="cuda") + 0.5
        flags = (torch.rand(shape, generator=g, device="cuda") < 0.1).to(torch.uint8)
        wl.spws.append(synth.SourceSpw(torch.as_tensor(uvw, device="cuda"), f, vis.to(torch.complex128) if wide else vis,
                                       wts, flags, 2e-4, -1e-4, z, None))
    return wl


WINDOWS = [(700, 40, 2, False), (33, 130, 4, False), (1, 33, 1, False), (2500, 64, 2, False), (300, 20, 2, True),
           (65, 100, 1, False), (900, 17, 4, False)]


@pytest.mark.parametrize("tuning", [None, dict(chans_per_lane=4), dict(sort_rows=0, chans_per_lane=2)])
@pytest.mark.parametrize("host,wave", [(False, 0), (True, 0), (True, 256 << 10)])
def test_classes_against_oracle(V, host, wave, tuning):
    wl = _workload(WINDOWS)
    for precision in (V.PREC_MIXED, V.PREC_FP64):
        st = V.Stack(wl.nu, wl.nv, wl.nrest, wl.npol, wl.du, wl.dv, rest_f0=wl.rest_f0, rest_df=wl.rest_df,
                     central_freq=wl.central_freq, precision=precision)
        try:
            st.set_tuning(**(tuning or {}))
            st.set_wave_bytes(wave)
            for again in range(3):   # planned, captured, replayed (device windows)
                st.zero()
                keep = []
                for s in wl.spws:
                    args = [s.uvw, s.freqs, s.vis, s.weights, s.flags]
                    if host:
                        args = [a.cpu().pin_memory() if isinstance(a, torch.Tensor) else a for a in args]
                    keep.append(args)
                    st.add_source(*args, l=s.l, m=s.m, z=s.z)
                st.run()
                g = {k: v.cpu().numpy() for k, v in st.read_cube(device=True, f64=True).items()}
            g["sum_wv"] = g["sum_wv"][..., 0] + 1j * g["sum_wv"][..., 1]
            g["stats"], g["lattice"] = st.stats(), st.lattice()
        finally:
            st.close()
        o = H.run_oracle(wl)
        H.compare(g, o, H.TOL_MIXED if precision == V.PREC_MIXED else H.TOL_FP64, what="%s %s %s" % (host, tuning, precision))
        assert g["stats"]["n_stacked"] > 0
