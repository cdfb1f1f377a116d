"""Performance cases: the calls that users of the stacking library make.

A case is a dict of plain values.  `kind` says which call it makes:

  stack    a whole stack on the device: zero the cube, queue every window
           (Stack.add_source), run, read the cube back to device tensors
  stream   the same from pinned host memory, with the touched entries only
           read back to the host (Stack.read_cube_sparse)
  regrid   the per-row output of one window (Stack.regrid_rows)
  contsub  continuum subtraction over a stacked cube (Stack.contsub)

The windows of a case are laid out by `shape_seed` (row counts, channel
counts, pols, redshifts, frequencies: a function of the case alone); the
antennas, source offsets, visibilities, weights and flags come from the seed
given to prepare().

  nsrc, nwin       sources, windows per source
  rows, uneven     rows per window: a fixed number, or a lognormal with that
                   median and sigma `uneven` (at most rows_max)
  nchan, npol      a number, or a text of numbers to choose from
  width            bandwidth of a window, Hz
  centres          observed centres (Hz) as a text, or "" for windows near
                   the line's observed frequency
  line             rest frequency of the cube's centre, Hz
  storage          c64, c128, f16, bf16
  pool             0, or complex values in a pool that the windows are views
                   of (more visibilities than a prepared state should hold)
  flags            largest flagged fraction (0: no flag arrays)
  nu, nrest, planes   cube cells per side, rest channels, planes
  coarse           rest channel width over the widest rest-frame input channel
                   (1: the library's own rule)
"""
import math

import numpy as np
import torch

from paper_2609_01897_gb300 import vista

C_LIGHT = 299792458.0
ARCSEC = math.pi / (180.0 * 3600.0)
CII = 1900.537e9          # [CII] 158 um
CO32 = 345.796e9          # CO(3-2)
CO109 = 1151.985452e9     # CO(10-9)
CO21 = 230.538e9          # CO(2-1)
HI = 1420.405752e6

_BASE = dict(kind="stack", nsrc=1, nwin=1, rows=1000, uneven=0.0, rows_max=200000, nchan=64, npol=2, width=1e9,
             centres="", descending=False, line=CO21, z_lo=1.0, z_hi=3.0, n_ant=30, radius=500.0, t_int=30.0,
             offset=10.0, storage="c64", pool=0, flags=0.01, nu=64, nrest=128, planes=2, coarse=1.0,
             nearest=False, fold=False, reproject=False, pol_map=False, fp64=False, order=1, shape_seed=1)


def _case(name, **kw):
    c = dict(_BASE, **kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # a test-sized stack: eight short windows, where latency and launches count
        _case("stack_tiny", nsrc=8, rows=900, nchan=64, width=1e9, n_ant=10, radius=250.0, nu=64, nrest=128),
        # one ordinary full-polarisation window into a small cube
        _case("stack_one_4pol", rows=10001, nchan=240, npol=4, width=1.875e9, flags=0.03, line=CII, z_lo=1.5, z_hi=2.5,
              nu=64, nrest=256, planes=4, shape_seed=2),
        # an ALMA compact-array survey: two windows a source, part of them in the cube's range
        _case("stack_alma", nsrc=24, nwin=2, rows=108360, nchan=120, width=1.875e9, centres="100e9,112e9", line=CO32,
              z_lo=2.0, z_hi=2.6, n_ant=43, nu=256, nrest=512, shape_seed=3),
        # an archive stack: uneven windows, 128 to 3840 channels, 2 or 4 pols, the widest dynamic range of bin widths
        _case("stack_archive", nsrc=48, nwin=2, rows=20000, uneven=1.0, rows_max=120000, nchan="128,240,480,960,3840",
              npol="2,4", width=1.875e9, line=CII, z_lo=0.5, z_hi=4.0, radius=2000.0, flags=0.1, pool=2 << 30, nu=256,
              nrest=1024, planes=4, shape_seed=4),
        # wideband HI: 4096 channels, half-precision storage, uv tracks that cross many cells along the band
        _case("stack_wideband_f16", nsrc=8, rows=40320, nchan=4096, width=856e6, centres="1284e6", line=HI, z_lo=0.1,
              z_hi=0.5, n_ant=64, radius=4000.0, t_int=8.0, storage="f16", nu=256, nrest=1024, shape_seed=5),
        # long baselines (large phases), bfloat16 storage, 960 channels
        _case("stack_long_bf16", nsrc=8, rows=54180, nchan=960, width=1.875e9, line=CO109, z_lo=2.0, z_hi=3.0, n_ant=43,
              radius=8000.0, offset=60.0, storage="bf16", nu=256, nrest=512, shape_seed=6),
        # ragged re-projected windows: odd sizes, descending axes, 1/2/4 pols with pol maps, Hermitian fold, nearest bin
        _case("stack_ragged", nsrc=12, rows=5003, uneven=0.8, rows_max=30000, nchan="33,65,117,250", npol="1,2,4",
              width=1.2e9, descending=True, radius=1500.0, offset=30.0, flags=0.05, nu=128, nrest=160, planes=4,
              nearest=True, fold=True, reproject=True, pol_map=True, shape_seed=7),
        # the FP64 form on double-precision visibilities
        _case("stack_fp64", nsrc=4, rows=18060, nchan=120, width=1.875e9, line=CO32, z_lo=2.0, z_hi=3.0, n_ant=43,
              storage="c128", nu=128, nrest=256, fp64=True, shape_seed=8),
        # windows in pinned host memory, streamed through the device; the touched entries back to the host
        _case("stream_host", kind="stream", nsrc=4, rows=21700, nchan=480, width=1.875e9, line=CII, z_lo=1.0, z_hi=3.0,
              n_ant=32, radius=1000.0, nu=96, nrest=512, shape_seed=9),
        # the per-row output of a wide full-polarisation window
        _case("regrid_wide_4pol", kind="regrid", rows=12000, nchan=3840, npol=4, width=1.875e9, line=CII, z_lo=1.0,
              z_hi=2.0, radius=2000.0, flags=0.03, nu=16, nrest=1024, planes=4, coarse=4.0, shape_seed=10),
        # the per-row output of a half-precision window whose channels are as wide as the rest channels
        _case("regrid_f16", kind="regrid", rows=27090, nchan=120, width=1.875e9, line=CO32, z_lo=2.0, z_hi=3.0, n_ant=43,
              storage="f16", nu=16, nrest=150, shape_seed=11),
        # continuum subtraction over an archive-sized cube, part of its uv cells touched
        _case("contsub_linear", kind="contsub", nsrc=4, rows=20000, nchan=960, npol=4, width=1.875e9, line=CII, z_lo=1.0,
              z_hi=3.0, radius=2000.0, flags=0.03, nu=256, nrest=1024, planes=4, order=1, shape_seed=12),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["stack"] * 6 + ["stream", "regrid", "regrid", "contsub"])
    npol = rng.choice([1, 2, 2, 4])
    c = _case("", kind=kind, npol=npol, planes=max(npol, 2), shape_seed=rng.randrange(1 << 20),
              line=rng.choice([CO21, CO32, CO109, CII]), storage=rng.choice(["c64", "c64", "c64", "f16", "bf16"]),
              width=rng.choice([0.5e9, 1e9, 1.875e9]), radius=float(_log(rng, 250, 8000)), n_ant=rng.randrange(8, 51),
              offset=rng.choice([5.0, 10.0, 60.0]), flags=rng.choice([0.0, 0.01, 0.05, 0.1]), z_lo=0.5,
              z_hi=rng.choice([1.0, 2.0, 4.0]), coarse=rng.choice([1.0, 1.0, 1.5, 6.0]), nearest=rng.random() < 0.2,
              fold=rng.random() < 0.25, descending=rng.random() < 0.25, nchan=_log(rng, 24, 3840))
    c["nrest"] = min(1024, max(48, int(c["nchan"] * rng.uniform(0.6, 1.6) / c["coarse"])))
    if kind == "regrid":
        c.update(nu=16, nearest=False, fold=False)
        c["rows"] = _log(rng, 500, min(100000, 2.0e8 / (max(c["nchan"], c["nrest"]) * npol)))
        return c
    if kind == "stack":
        c["reproject"] = rng.random() < 0.2
        c["fp64"] = rng.random() < 0.12
        if c["fp64"]:
            c["storage"] = rng.choice(["c64", "c128"])
    # visibilities of the stack, shared among its sources, and a cube to match
    total = _log(rng, 2e6, 6e7 if c["fp64"] else 1.2e8 if kind == "stream" else 1e9)
    c.update(nsrc=_log(rng, 1, 24), uneven=rng.choice([0.0, 0.5, 1.0]))
    c["rows"] = int(max(2, min(100000, total / (c["nsrc"] * c["nchan"] * npol))))
    c["rows_max"] = 4 * c["rows"]
    most = math.sqrt(min(2e8, total) / (c["nrest"] * c["planes"]))
    c["nu"] = 2 * max(8, min(128, int(0.5 * most * rng.uniform(0.3, 1.0))))
    if kind == "contsub":
        c.update(order=rng.choice([0, 1, 1, 2]), nearest=False)
    return c


# ------------------------------------------------------------------ layout

def _pick(rng, v):
    return int(v) if not isinstance(v, str) else int(rng.choice([int(x) for x in v.split(",")]))


def _layout(c):
    """The windows of a case (a function of the case alone): dicts with the
    source, rows, channel frequencies, pols, redshift and pol map."""
    rng = np.random.default_rng(c["shape_seed"])
    centres = [float(x) for x in c["centres"].split(",")] if c["centres"] else []
    wins = []
    for s in range(c["nsrc"]):
        z = float(rng.uniform(c["z_lo"], c["z_hi"]))
        rows = c["rows"]
        if c["uneven"]:
            rows = int(round(rng.lognormal(math.log(c["rows"]), c["uneven"])))
        rows = max(1, min(rows, c["rows_max"]))
        npol = _pick(rng, c["npol"])
        for k in range(c["nwin"]):
            nchan = _pick(rng, c["nchan"])
            near = c["line"] / (1.0 + z) + float(rng.uniform(-0.4, 0.4)) * c["width"]
            fc = centres[k % len(centres)] if centres else near
            df = c["width"] / nchan
            f = fc - 0.5 * (nchan - 1) * df + np.arange(nchan, dtype=np.float64) * df
            if c["descending"] and s % 2:
                f = np.ascontiguousarray(f[::-1])
            pm = None
            if c["pol_map"]:
                pm = np.array([(s + p) % c["planes"] for p in range(npol)], dtype=np.int32)
                if npol > 1:
                    pm[-1] = -1
            wins.append(dict(source=s, rows=rows, freqs=f, df=df, npol=npol, z=z, pol_map=pm))
    return wins


def _lattice(c, wins):
    """The common rest lattice: `coarse` times the widest rest-frame channel, centred on the line."""
    df = max(w["df"] * (1.0 + w["z"]) for w in wins) * c["coarse"]
    return c["line"] - 0.5 * c["nrest"] * df, df


def _cell(c, wins):
    """The uv cell size (wavelengths): the longest possible baseline just fits."""
    return 2.0 * 1.0001 * 2.0 * c["radius"] * max(float(w["freqs"].max()) for w in wins) / C_LIGHT / c["nu"]


def _bins(c, w, f0, df):
    """Weights of the window's channels on the rest lattice, [nchan, nrest] float64."""
    f = w["freqs"]
    zf = 1.0 + w["z"]
    if c["nearest"]:
        j = np.floor((f * zf - f0) / df).astype(np.int64)
        W = np.zeros((f.size, c["nrest"]))
        ok = (j >= 0) & (j < c["nrest"])
        W[np.nonzero(ok)[0], j[ok]] = 1.0
        return W
    d = np.abs(np.gradient(f))
    lo, hi = ((f - 0.5 * d) * zf)[:, None], ((f + 0.5 * d) * zf)[:, None]
    e = f0 + df * np.arange(c["nrest"] + 1)[None, :]
    return np.maximum(0.0, np.minimum(hi, e[:, 1:]) - np.maximum(lo, e[:, :-1])) / (hi - lo)


# ------------------------------------------------------------------ inputs

def _tracks(rng, c, rows):
    """uvw (metres) of the first `rows` rows of an Earth-rotation track, time-major, float64."""
    r = c["radius"] * np.sqrt(rng.random(c["n_ant"]))
    a = 2.0 * np.pi * rng.random(c["n_ant"])
    east, north = r * np.cos(a), r * np.sin(a)
    i, j = np.triu_indices(c["n_ant"], k=1)
    lat, dec = math.radians(-23.0), math.radians(-30.0)
    y = east[j] - east[i]
    x, zz = -math.sin(lat) * (north[j] - north[i]), math.cos(lat) * (north[j] - north[i])
    nt = (rows + i.size - 1) // i.size
    ha = rng.uniform(-1.0, 1.0) + (np.arange(nt) - 0.5 * nt) * c["t_int"] * (2.0 * np.pi / 86164.0905)
    sh, ch = np.sin(ha)[:, None], np.cos(ha)[:, None]
    u = sh * x + ch * y
    v = -math.sin(dec) * (ch * x - sh * y) + math.cos(dec) * zz
    w = math.cos(dec) * (ch * x - sh * y) + math.sin(dec) * zz
    return np.ascontiguousarray(np.stack([u, v, w], -1).reshape(-1, 3)[:rows])


def _turns(uvw, l, m, freqs):
    """Turns of the phase tau nu / c, [nrow, nchan] float64."""
    tau = uvw[:, 0] * l + uvw[:, 1] * m + uvw[:, 2] * (math.sqrt(1.0 - l * l - m * m) - 1.0)
    return tau[:, None] * (torch.as_tensor(freqs, device=uvw.device) / C_LIGHT)[None, :]


def _visibilities(g, uvw, w, l, m, storage):
    """A faint point source with a line, under noise, [nrow, nchan, npol] of the
    storage type, and the scale of the 16-bit types."""
    f = w["freqs"]
    shape = (uvw.shape[0], f.size, w["npol"])
    vis = torch.complex(torch.randn(shape, generator=g, device="cuda"), torch.randn(shape, generator=g, device="cuda"))
    amp = torch.as_tensor(0.1 + 0.2 * np.exp(-0.5 * ((np.arange(f.size) - 0.5 * f.size) / (0.05 * f.size + 1)) ** 2),
                          device="cuda", dtype=torch.float32)
    step = max(1, (1 << 25) // f.size)
    for r in range(0, shape[0], step):
        t = _turns(uvw[r:r + step], l, m, f)
        ph = (-2.0 * math.pi * (t - torch.floor(t))).float()
        vis[r:r + step] += torch.polar(amp[None, :].expand_as(ph), ph)[:, :, None]
    vis *= 1e-3
    if storage == "c64":
        return vis, 1.0
    if storage == "c128":
        return vis.to(torch.complex128), 1.0
    pairs = torch.view_as_real(vis)
    e = math.ceil(math.log2(float(pairs.abs().max())))
    scale = 2.0 ** (e - 15) if storage == "f16" else 2.0 ** e
    return (pairs / scale).to(torch.float16 if storage == "f16" else torch.bfloat16), scale


def _inputs(c, seed):
    """Device arrays of every window: lists of (window, uvw, vis, weights,
    flags, l, m, scale, reproject)."""
    wins = _layout(c)
    rng = np.random.default_rng([seed, c["shape_seed"]])
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    pool = fpool = None
    if c["pool"]:
        pool = torch.empty(c["pool"], dtype=torch.complex64, device="cuda")
        torch.view_as_real(pool).normal_(generator=g)
        fpool = torch.empty(c["pool"], dtype=torch.uint8, device="cuda")
        part = c["pool"] // 16
        for k in range(16):
            fpool[k * part:(k + 1) * part] = torch.rand(part, generator=g, device="cuda") < c["flags"] * k / 15.0
    out, last = [], None
    for w in wins:
        if w["source"] != last:
            last = w["source"]
            uvw = torch.as_tensor(_tracks(rng, c, w["rows"]), device="cuda")
            l, m = (float(x) for x in rng.uniform(-c["offset"], c["offset"], 2) * ARCSEC)
            wts = torch.rand((w["rows"], w["npol"]), generator=g, device="cuda") + 0.5
            rep = None
            if c["reproject"]:
                ra0, dec0 = 0.3 + 0.01 * w["source"], math.radians(-30.0)
                rep = (ra0, dec0, ra0 + l / math.cos(dec0), dec0 + m)
                l, m = _offset(rep)
        shape = (w["rows"], w["freqs"].size, w["npol"])
        n = shape[0] * shape[1] * shape[2]
        if pool is not None:
            o = int(rng.integers(0, (c["pool"] - n) // 16 + 1)) * 16
            fo = int(rng.integers(0, (c["pool"] - n) // 16 + 1)) * 16
            vis, scale, flags = pool[o:o + n].view(shape), 1.0, fpool[fo:fo + n].view(shape)
        else:
            vis, scale = _visibilities(g, uvw, w, l, m, c["storage"])
            frac = c["flags"] * float(rng.uniform(0.2, 1.0))
            flags = (torch.rand(shape, generator=g, device="cuda") < frac).to(torch.uint8) if c["flags"] else None
        out.append((w, uvw, vis, wts, flags, l, m, scale, rep))
    return out


def _offset(rep):
    """Direction cosines of (ra1, dec1) seen from (ra0, dec0)."""
    ra0, dec0, ra1, dec1 = rep
    return (math.cos(dec1) * math.sin(ra1 - ra0),
            math.sin(dec1) * math.cos(dec0) - math.cos(dec1) * math.sin(dec0) * math.cos(ra1 - ra0))


def _stack(c, wins, fixed):
    f0, df = _lattice(c, wins)
    du = _cell(c, wins)
    kw = dict(rest_f0=f0, rest_df=df) if fixed else dict(central_freq=c["line"])
    return vista.Stack(c["nu"], c["nu"], c["nrest"], c["planes"], du, du,
                       bin_mode=vista.BIN_NEAREST if c["nearest"] else vista.BIN_OVERLAP,
                       precision=vista.PREC_FP64 if c["fp64"] else vista.PREC_MIXED, hermitian_fold=c["fold"], **kw)


def _queue(st, args):
    for w, uvw, vis, wts, flags, l, m, scale, rep in args:
        st.add_source(uvw, w["freqs"], vis, wts, flags, l=l, m=m, z=w["z"], pol_map=w["pol_map"], vis_scale=scale,
                      reproject=rep)


def _line_free(c):
    lf = np.ones(c["nrest"], dtype=bool)
    lf[int(0.4 * c["nrest"]):int(0.6 * c["nrest"])] = False
    return lf


def prepare(case, seed):
    c = case
    args = _inputs(c, seed)
    wins = [a[0] for a in args]
    st = _stack(c, wins, fixed=c["kind"] == "regrid" or c["coarse"] != 1.0)
    state = {"case": c, "stack": st, "args": args}
    if c["kind"] == "stream":
        state["args"] = [(w, *[None if t is None else t.cpu().pin_memory() for t in (uvw, vis, wts, flags)], *rest)
                         for w, uvw, vis, wts, flags, *rest in args]
        # host buffers as large as the cube, kept for every stack, as such a program would
        n = c["nu"] * c["nu"] * c["nrest"] * c["planes"]
        state["out"] = {k: torch.zeros(shape, dtype=dt).pin_memory() for k, shape, dt in (
            ("index", n, torch.int64), ("sum_wv", (n, 2), torch.float32), ("sum_w", n, torch.float32),
            ("sum_wvv", n, torch.float32), ("count", n, torch.int32))}
    elif c["kind"] == "contsub":
        _queue(st, args)
        st.run()
        st.stats()
        state["args"] = None
        state["line_free"] = _line_free(c)
    elif c["kind"] == "regrid":
        state["args"] = args[0]
    return state


def run(state):
    c, st = state["case"], state["stack"]
    if c["kind"] == "regrid":
        w, uvw, vis, _, flags, l, m, scale, _ = state["args"]
        out_vis, wsum, _ = st.regrid_rows(uvw, w["freqs"], vis, flags, l=l, m=m, z=w["z"], vis_scale=scale)
        return {"vis": out_vis, "wsum": wsum}
    if c["kind"] == "contsub":
        return st.contsub(state["line_free"], order=c["order"])
    st.zero()
    _queue(st, state["args"])
    st.run()
    if c["kind"] == "stream":
        st.read_cube_sparse(out=state["out"])   # the first n entries of each buffer
        return state["out"]
    return st.read_cube(f64=c["fp64"])


# -------------------------------------------------------------------- work

_VALUE = {"c64": 8, "c128": 16, "f16": 4, "bf16": 4}


def _in_cube(c, wins):
    """Per window: the channels that reach the rest lattice."""
    f0, df = _lattice(c, wins)
    top = f0 + c["nrest"] * df
    got = []
    for w in wins:
        half = 0.0 if c["nearest"] else 0.5 * w["df"]
        lo, hi = (w["freqs"] - half) * (1.0 + w["z"]), (w["freqs"] + half) * (1.0 + w["z"])
        got.append(int(np.sum((hi > f0) & (lo < top))))
    return got


def work(case):
    c = case
    wins = _layout(c)
    n = c["nu"] * c["nu"] * c["nrest"] * c["planes"]
    one = _VALUE[c["storage"]] + (1 if c["flags"] else 0)
    if c["kind"] == "contsub":
        return {"bytes": n * 20.0, "flops": n * 12.0}
    used = _in_cube(c, wins)
    nvis = sum(float(w["rows"]) * k * w["npol"] for w, k in zip(wins, used))
    rows = sum(w["rows"] * (24.0 + 4.0 * w["npol"]) for w, k in zip(wins, used) if k)
    if c["kind"] == "regrid":
        w = wins[0]
        return {"bytes": nvis * one + w["rows"] * (24.0 + 12.0 * c["nrest"] * w["npol"]), "flops": nvis * 22.0}
    # the dense cube comes back in full, the sparse one at its 28 bytes per touched entry (a few % of the input)
    back = 0.0 if c["kind"] == "stream" else n * (36.0 if c["fp64"] else 20.0)
    return {"bytes": nvis * one + rows + back, "flops": nvis * 22.0}


# ------------------------------------------------------------------- exact

def _complex128(vis, scale):
    if vis.is_complex():
        return vis.to(torch.complex128)
    return torch.view_as_complex(vis.double() * scale)


def _rotated(uvw, rep):
    """u, v for the new phase centre."""
    ra0, dec0, ra1, dec1 = rep

    def frame(ra, dec):
        return np.array([[-math.sin(ra), math.cos(ra), 0.0],
                         [-math.sin(dec) * math.cos(ra), -math.sin(dec) * math.sin(ra), math.cos(dec)],
                         [math.cos(dec) * math.cos(ra), math.cos(dec) * math.sin(ra), math.sin(dec)]])

    R = frame(ra1, dec1) @ frame(ra0, dec0).T
    return [(R[i, 0] * uvw[:, 0] + R[i, 1] * uvw[:, 1]) + R[i, 2] * uvw[:, 2] for i in (0, 1)]


def _exact_cube(c, seed):
    """The cube's sums in 64 bits, [entries, 4] = (re, im, weight, |V|^2), and counts."""
    args = _inputs(c, seed)
    wins = [a[0] for a in args]
    f0, df = _lattice(c, wins)
    scale_uv = 1.0 / (C_LIGHT * _cell(c, wins))
    nu, nrest, planes = c["nu"], c["nrest"], c["planes"]
    cube = torch.zeros((nu * nu * nrest * planes, 4), dtype=torch.float64, device="cuda")
    count = torch.zeros(nu * nu * nrest * planes, dtype=torch.int32, device="cuda")
    for w, uvw, vis, wts, flags, l, m, scale, rep in args:
        W = _bins(c, w, f0, df)
        chans = np.nonzero(W.any(axis=1))[0]
        if not chans.size:
            continue
        k0, k1 = int(chans[0]), int(chans[-1]) + 1
        first = torch.as_tensor(np.argmax(W[k0:k1] > 0, axis=1), device="cuda")
        nb = int((W > 0).sum(axis=1).max())
        Wd = torch.as_tensor(W[k0:k1], device="cuda")
        s = torch.as_tensor(w["freqs"][k0:k1] * scale_uv, device="cuda")
        u, v = (uvw[:, 0], uvw[:, 1]) if rep is None else _rotated(uvw, rep)
        step = max(1, (1 << 24) // (k1 - k0))
        for r in range(0, w["rows"], step):
            ur, vr = u[r:r + step], v[r:r + step]
            t = _turns(uvw[r:r + step], l, m, w["freqs"][k0:k1])
            ph = torch.polar(torch.ones_like(t), 2.0 * math.pi * (t - torch.floor(t)))
            conj = torch.zeros_like(ur, dtype=torch.bool)
            if c["fold"]:
                conj = (vr < 0) | ((vr == 0) & (ur < 0))
                ur, vr = torch.where(conj, -ur, ur), torch.where(conj, -vr, vr)
            iu = torch.floor(ur[:, None] * s[None, :]).long() + nu // 2
            iv = torch.floor(vr[:, None] * s[None, :]).long() + nu // 2
            on = (iu >= 0) & (iu < nu) & (iv >= 0) & (iv < nu)
            cell = iv * nu + iu
            x = _complex128(vis[r:r + step, k0:k1], scale)
            for p in range(w["npol"]):
                plane = p if w["pol_map"] is None else int(w["pol_map"][p])
                if plane < 0:
                    continue
                ok = on if flags is None else on & (flags[r:r + step, k0:k1, p] == 0)
                V = x[:, :, p] * ph
                im = torch.where(conj[:, None], -V.imag, V.imag)
                a2 = x[:, :, p].real ** 2 + x[:, :, p].imag ** 2
                wr = wts[r:r + step, p].double()[:, None]
                val = torch.stack([wr * V.real, wr * im, wr.expand_as(a2), wr * a2], -1)
                for b in range(nb):
                    j = torch.clamp(first + b, max=nrest - 1)
                    ww = torch.where(first + b < nrest, Wd.gather(1, j[:, None])[:, 0], torch.zeros_like(Wd[:, 0]))
                    use = ok & (ww > 0)[None, :]
                    idx = ((cell * nrest + j[None, :]) * planes + plane)[use]
                    cube.index_add_(0, idx, (val * ww[None, :, None])[use])
                    count.index_add_(0, idx, torch.ones_like(idx, dtype=torch.int32))
    return cube, count


def _exact_contsub(c, cube):
    """The sums less the weighted polynomial fit of every (cell, plane)."""
    nrest, planes = c["nrest"], c["planes"]
    x = torch.as_tensor((2.0 * np.arange(nrest) - (nrest - 1)) / nrest, device="cuda")
    lf = torch.as_tensor(_line_free(c), device="cuda")
    cube = cube.view(-1, nrest, planes, 4)
    out = torch.empty(cube.shape[:3] + (2,), dtype=torch.float64, device="cuda")
    step = max(1, (1 << 24) // (nrest * planes))
    for a in range(0, cube.shape[0], step):
        part = cube[a:a + step]
        w = part[..., 2]
        fit = lf[None, :, None] & (w > 0)
        nfit = fit.sum(1)
        res = part[..., :2].clone()
        wf = torch.where(fit, w, torch.zeros_like(w))
        yf = torch.where(fit[..., None], part[..., :2], torch.zeros_like(part[..., :2]))
        pw = torch.stack([x ** k for k in range(2 * c["order"] + 1)])
        M = torch.einsum("nj,cjp->cpn", pw, wf)
        B = torch.einsum("nj,cjpr->cpnr", pw[:c["order"] + 1], yf)
        for d in range(c["order"] + 1):
            at = torch.nonzero((nfit - 1 == d) | ((nfit - 1 > d) if d == c["order"] else torch.zeros_like(nfit, dtype=torch.bool)))
            if not at.shape[0]:
                continue
            i, p = at[:, 0], at[:, 1]
            A = torch.stack([M[i, p, k:k + d + 1] for k in range(d + 1)], 1)
            coef = torch.linalg.solve(A, B[i, p, :d + 1])
            model = torch.einsum("nj,snr->sjr", pw[:d + 1], coef)
            res[i, :, p] -= w[i, :, p][..., None] * model
        out[a:a + step] = res
    return out.view(c["nu"], c["nu"], nrest, planes, 2)


def _exact_regrid(c, seed):
    w, uvw, vis, _, flags, l, m, scale, _ = _inputs(c, seed)[0]
    f0, df = _lattice(c, [w])
    W = torch.as_tensor(_bins(c, w, f0, df), device="cuda")
    shape = (w["rows"], c["nrest"], w["npol"])
    out = torch.zeros(shape, dtype=torch.complex128, device="cuda")
    wsum = torch.zeros(shape, dtype=torch.float64, device="cuda")
    step = max(1, (1 << 23) // w["freqs"].size)
    for r in range(0, w["rows"], step):
        t = _turns(uvw[r:r + step], l, m, w["freqs"])
        ph = torch.polar(torch.ones_like(t), 2.0 * math.pi * (t - torch.floor(t)))
        for p in range(w["npol"]):
            V = _complex128(vis[r:r + step, :, p], scale) * ph
            ok = torch.ones_like(t) if flags is None else (flags[r:r + step, :, p] == 0).double()
            ws = ok @ W
            den = torch.where(ws > 0, ws, torch.ones_like(ws))
            out[r:r + step, :, p] = torch.complex((V.real * ok) @ W / den, (V.imag * ok) @ W / den)
            wsum[r:r + step, :, p] = ws
    return {"vis": out, "wsum": wsum}


def exact(case, seed):
    c = case
    if c["pool"]:
        return None   # billions of visibilities: too long in 64 bits
    if c["kind"] == "regrid":
        return _exact_regrid(c, seed)
    cube, count = _exact_cube(c, seed)
    if c["kind"] == "contsub":
        return _exact_contsub(c, cube)
    if c["kind"] == "stream":
        at = torch.nonzero(count)[:, 0]
        out = torch.zeros_like(cube)
        out[:at.shape[0]] = cube[at]
        return {"index": None, "sum_wv": out[:, :2], "sum_w": out[:, 2], "sum_wvv": out[:, 3], "count": None}
    shape = (c["nu"], c["nu"], c["nrest"], c["planes"])
    return {"sum_wv": cube[:, :2].reshape(shape + (2,)), "sum_w": cube[:, 2].reshape(shape),
            "sum_wvv": cube[:, 3].reshape(shape), "count": None}
