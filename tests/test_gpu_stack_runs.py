"""How the stacking kernel ends runs, against the FP64 oracle at the edges of
its branches: a rest bin wider or narrower than a channel (runs merged over
neighbouring channels, a chunk in one or two bins, channels that reach three
bins), ascending and descending axes, irregular plane maps, the Hermitian
fold, odd channel counts and item sizes."""
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


def _workload(npol, coarse, descending, pol_map, nrow, nchan):
    from paper_2609_01897_gb300 import synth
    rng = np.random.default_rng([npol, int(10 * coarse), nrow, nchan])
    df, line, z = 2e6, 230e9, 0.7
    f = (line / (1 + z)) + df * (np.arange(nchan) - 0.5 * nchan)
    if descending:
        f = f[::-1].copy()
    # tracks that stay in a cell for a few rows and cross cell edges inside the band
    t = np.arange(nrow)
    uvw = np.stack([300.0 * np.sin(0.011 * t + 0.3), 240.0 * np.cos(0.017 * t), 40.0 * np.sin(0.01 * t)], 1)
    uvw *= np.where(rng.random(nrow) < 0.1, -1.0, 1.0)[:, None]
    g = torch.Generator(device="cuda")
    g.manual_seed(nrow)
    shape = (nrow, nchan, npol)
    vis = torch.complex(torch.randn(shape, generator=g, device="cuda"), torch.randn(shape, generator=g, device="cuda"))
    wts = torch.rand((nrow, npol), generator=g, device="cuda") + 0.5
    flags = (torch.rand(shape, generator=g, device="cuda") < 0.1).to(torch.uint8)
    s = synth.SourceSpw(torch.as_tensor(uvw, device="cuda"), f, vis, wts, None if descending else flags, 2e-4, -1e-4, z,
                        None if pol_map is None else np.array(pol_map, dtype=np.int32))
    rest_df = df * (1 + z) * coarse
    nrest = max(2, int(1.1 * nchan / coarse))
    du = 2 * 330.0 * f.max() / H.C_LIGHT / 24
    return synth.Workload("runs", 24, 24, nrest, 4, du, du, line, [s], rest_df=rest_df, rest_f0=line - 0.45 * nrest * rest_df)


MAPS = {1: [None, [3]], 2: [None, [2, 3], [1, 2]], 4: [None, [3, 2, -1, 0]]}


@pytest.mark.parametrize("nrow,nchan,tuning", [
    (1, 33, None), (2, 64, dict(rows_per_item=1)), (65, 31, dict(rows_per_item=31)), (97, 70, dict(rows_per_item=33)),
    (300, 96, dict(chans_per_lane=2)), (257, 130, dict(rows_per_item=256, chans_per_lane=4, prefetch_rows=8)),
    (128, 32, dict(prefetch_rows=2))])
@pytest.mark.parametrize("coarse", [0.4, 1.0, 1.37, 5.0, 60.0])
@pytest.mark.parametrize("npol", [1, 2, 4])
def test_runs_against_oracle(V, npol, coarse, nrow, nchan, tuning):
    for k, pm in enumerate(MAPS[npol]):
        for descending in (False, True):
            wl = _workload(npol, coarse, descending, pm, nrow, nchan)
            fold = (k + descending) % 2 == 1
            g = H.run_gpu(wl, fold=fold, tuning=tuning)
            o = H.run_oracle(wl, fold=fold)
            H.compare(g, o, H.TOL_MIXED, what="%s %s %s" % (pm, descending, fold))
            H.stats_equal(g, o)
            assert g["stats"]["n_stacked"] > 0
