"""The processing order of rows inside a uv cell: by the part of the cell they
lie in, where 32 rows alternate between parts more than twice as often as they
must, else in row order.  The order is compared with a NumPy restatement, and
the stack with the FP64 oracle, at ragged row counts, over windows that share a
warp, folded and not, and for coordinates off the grid."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

from tests import gpu_helpers as H  # noqa: E402

NU, NCHAN, LINE, Z, DF = 16, 24, 230e9, 0.7, 40e6


@pytest.fixture(scope="module")
def V():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_01897_gb300 import build
    build.build()
    from paper_2609_01897_gb300 import vista
    vista.lib()
    return vista


def _workload(kind, rows):
    from paper_2609_01897_gb300 import synth
    f = LINE / (1 + Z) + DF * (np.arange(NCHAN) - 0.5 * NCHAN)
    half = 300.0
    du = 2 * half * f.max() / H.C_LIGHT / NU
    wl = synth.Workload(kind, NU, NU, 64, 2, du, du, LINE, [], rest_df=DF * (1 + Z), rest_f0=LINE - 32 * DF * (1 + Z))
    for k, n in enumerate(rows):
        rng = np.random.default_rng([n, k])
        if kind == "scattered":      # a few cells, rows anywhere in them
            xy = rng.uniform(-1.4, 1.4, (n, 2)) * 2 * half / NU
        elif kind == "tracks":       # slow tracks: row order is kept
            t = np.arange(n)[:, None] * 2e-4 + np.array([[0.1, 0.7]])
            xy = 220.0 * np.sin(t)
        else:                        # both, some far off the grid
            t = np.arange(n)[:, None] * 3e-4 + np.array([[0.1, 0.7]])
            xy = np.where(rng.random((n, 1)) < 0.5, 220.0 * np.sin(t), rng.uniform(-1.1, 1.1, (n, 2)) * half * rng.choice([0.2, 1.5]))
        uvw = np.concatenate([xy, rng.uniform(-30, 30, (n, 1))], 1)
        g = torch.Generator(device="cuda")
        g.manual_seed(n + k)
        shape = (n, NCHAN, 2)
        vis = torch.complex(torch.randn(shape, generator=g, device="cuda"), torch.randn(shape, generator=g, device="cuda"))
        wts = torch.rand((n, 2), generator=g, device="cuda") + 0.5
        flags = (torch.rand(shape, generator=g, device="cuda") < 0.1).to(torch.uint8)
        wl.spws.append(synth.SourceSpw(torch.as_tensor(uvw, device="cuda"), f, vis, wts, flags, 2e-4, -1e-4, Z, None))
    return wl


def _expected(wl, fold):
    """Per window, the rows in processing order; and the numbers of 32-row
    groups reordered and kept."""
    win, row, x, y = [], [], [], []
    for k, s in enumerate(wl.spws):
        u, v = (s.uvw.cpu().numpy()[:, i] for i in (0, 1))
        sign = np.where((v < 0) | ((v == 0) & (u < 0)), -1.0, 1.0) if fold else np.ones(len(u))
        su = np.float32(s.freqs[NCHAN // 2] * (1.0 / (H.C_LIGHT * wl.du)))
        xs, ys = (u * sign).astype(np.float32) * su, (v * sign).astype(np.float32) * su
        iu, iv = (np.clip(np.floor(c) + NU // 2, 0, NU - 1) for c in (xs, ys))
        o = np.lexsort((np.arange(len(u)), iu, iv))
        win += [k] * len(u)
        row += list(o)
        x += list(xs[o])
        y += list(ys[o])
    win, row, x, y = np.array(win), np.array(row), np.array(x, np.float32), np.array(y, np.float32)
    cx, cy = np.floor(x), np.floor(y)
    col = np.minimum(((x - cx) * np.float32(3)).astype(int), 2)
    part = 2 * col + ((y - cy >= 0.5).astype(int) ^ ((cx.astype(int) + col) & 1))
    moved = kept = 0
    for t in range(0, len(row), 32):
        e = slice(t, t + 32)
        head = np.ones(len(row[e]), bool)
        head[1:] = (np.diff(win[e]) != 0) | (np.diff(cx[e]) != 0) | (np.diff(cy[e]) != 0)
        p, cell = part[e], np.cumsum(head)
        T = int(((p[1:] != p[:-1]) & ~head[1:]).sum())
        G = len(np.unique(cell * 8 + p)) - int(head.sum())
        if T > 2 * G:
            row[e] = row[e][np.lexsort((np.arange(len(p)), p, cell))]
            moved += 1
        else:
            kept += 1
    return [row[win == k] for k in range(len(wl.spws))], moved, kept


@pytest.mark.parametrize("rows", [(1,), (31,), (33, 2), (64,), (1000, 31, 517), (2500, 700)])
@pytest.mark.parametrize("kind", ["scattered", "tracks", "both"])
@pytest.mark.parametrize("fold", [False, True])
def test_order_inside_cells(V, kind, rows, fold):
    wl = _workload(kind, rows)
    want, moved, kept = _expected(wl, fold)
    if sum(rows) > 1000:
        assert moved > kept if kind == "scattered" else kept > 0
    st = V.Stack(wl.nu, wl.nv, wl.nrest, wl.npol, wl.du, wl.dv, rest_f0=wl.rest_f0, rest_df=wl.rest_df,
                 central_freq=wl.central_freq, hermitian_fold=fold)
    try:
        for s in wl.spws:
            st.add_source(s.uvw, s.freqs, s.vis, s.weights, s.flags, l=s.l, m=s.m, z=s.z)
        st.run()
        for k, n in enumerate(rows):
            assert np.array_equal(st.debug_order(k, n).cpu().numpy(), want[k]), (kind, k)
    finally:
        st.close()
    g, o = H.run_gpu(wl, fold=fold), H.run_oracle(wl, fold=fold)
    H.compare(g, o, H.TOL_MIXED, what=kind)
    H.stats_equal(g, o)
