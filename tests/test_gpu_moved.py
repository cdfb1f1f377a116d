"""The mixed cube's masters are read and zeroed only where sums have been moved
into them: dense and sparse readback, continuum subtraction and zeroing after
stacks deep enough for checkpoints, with and without a fold, against the FP64
form on the same windows; cubes of odd sizes (the last word of bits is partial),
and other data stacked into the zeroed cube."""
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


def _window(seed, nrow, nchan, npol, half):
    rng = np.random.default_rng(seed)
    f = 135e9 + 2e6 * (np.arange(nchan) - 0.5 * nchan)
    uvw = np.concatenate([rng.uniform(-half, half, (nrow, 2)), rng.uniform(-20, 20, (nrow, 1))], 1)
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    shape = (nrow, nchan, npol)
    vis = torch.complex(torch.randn(shape, generator=g, device="cuda"), torch.randn(shape, generator=g, device="cuda"))
    wts = torch.rand((nrow, npol), generator=g, device="cuda") + 0.5
    flags = (torch.rand(shape, generator=g, device="cuda") < 0.05).to(torch.uint8)
    return torch.as_tensor(uvw, device="cuda"), f, vis, wts, flags


@pytest.mark.parametrize("nu,nrest,planes,nrow,nchan", [(4, 7, 1, 300, 9), (6, 33, 2, 3000, 64), (4, 5, 3, 9000, 33),
                                                        (10, 61, 4, 4000, 40)])
@pytest.mark.parametrize("runs", [1, 3])
def test_moved_masters(V, nu, nrest, planes, nrow, nchan, runs):
    npol = min(planes, 2) if planes != 4 else 4
    half, z = 40.0, 0.7
    du = 2 * half * 135.1e9 / H.C_LIGHT / (0.7 * nu)   # some cells stay untouched
    kw = dict(rest_f0=135e9 * (1 + z) - 0.5 * nrest * 2e6 * (1 + z), rest_df=2e6 * (1 + z), central_freq=135e9 * (1 + z))
    st = [V.Stack(nu, nu, nrest, planes, du, du, precision=p, **kw) for p in (V.PREC_MIXED, V.PREC_FP64)]
    free = np.ones(nrest, dtype=bool)
    free[nrest // 2] = False
    try:
        for cycle in range(3):   # other rows, and fewer of them, each time
            data = [_window(10 * cycle + k, nrow // (1 + cycle), nchan, npol, half / (1 + cycle)) for k in range(runs)]
            got = []
            for s in st:
                for u, f, v, w, fl in data:
                    s.add_source(u, f, v, w, fl, l=2e-4, m=-1e-4, z=z)
                    s.run()
                c = s.read_cube(device=True, f64=True)
                sp = s.read_cube_sparse()
                got.append(({k: x.cpu().numpy() for k, x in c.items()}, sp, s.contsub(free, 1).cpu().numpy()))
                s.zero()
                e = s.read_cube(device=True, f64=True)
                assert not any(x.any() for x in e.values())
            (m, ms, mc), (r, _, rc) = got
            assert np.array_equal(m["count"], r["count"]) and m["count"].sum() > 0
            scale = {"sum_w": r["sum_w"], "sum_wvv": r["sum_wvv"],
                     "sum_wv": np.sqrt(r["sum_w"] * r["sum_wvv"])[..., None]}   # >= sum w |V|
            for k, sc in scale.items():
                assert (np.abs(m[k] - r[k]) <= H.TOL_MIXED * sc + 1e-30).all(), k
            # the sparse form is the dense one at the touched entries
            idx = ms["index"].cpu().numpy() if torch.is_tensor(ms["index"]) else ms["index"]
            assert np.array_equal(np.sort(idx), np.flatnonzero(m["count"].reshape(-1)))
            w = ms["sum_w"].cpu().numpy() if torch.is_tensor(ms["sum_w"]) else ms["sum_w"]
            assert np.allclose(w, m["sum_w"].reshape(-1)[idx], rtol=2e-7, atol=0)
            sc = np.sqrt(r["sum_w"] * r["sum_wvv"])
            top = np.maximum(sc.max(), 1e-30)
            assert np.abs(mc - rc).max() <= 1e-4 * top
    finally:
        for s in st:
            s.close()
