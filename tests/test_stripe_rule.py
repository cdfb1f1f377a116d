"""The row ordering's stripes (host rule, no GPU): a small cube is cut into 32 for
a few windows, so that their sort fills the chip, and into ever fewer as the windows
grow in number, so that the buckets, a block and its tables each, stay near eight a
SM; and the layout's limits hold for any cube."""
import ctypes as C
import os
import random
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2609_01897_gb300", "csrc")


@pytest.fixture(scope="module")
def L(tmp_path_factory):
    d = tmp_path_factory.mktemp("stripes")
    src, so = os.path.join(d, "s.cpp"), os.path.join(d, "s.so")
    with open(src, "w") as f:
        f.write('#include "vista_internal.h"\n'
                'extern "C" int layout(int nu, int nv, int nrest, int npol, long long windows, int *o) {\n'
                '    return vista::stripe_layout(nu, nv, nrest, npol, vista::min_stripes(windows, (long long)nu * nv), o, o + 1, o + 2, o + 3);\n}\n'
                'extern "C" int limits(int *o) { o[0] = vista::MAX_LOCAL_KEYS; o[1] = vista::MAX_STRIPES; return 0; }\n')
    from paper_2609_01897_gb300 import build
    cuda = os.path.join(os.path.dirname(os.path.dirname(build._nvcc())), "include")
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I" + CSRC, "-I" + os.path.join(ROOT, "include"),
                           "-I" + cuda, src, "-o", so])
    return C.CDLL(so)


def _layout(L, nu, nv, nrest, npol, windows):
    o = (C.c_int * 4)()
    ok = L.layout(nu, nv, nrest, npol, C.c_longlong(windows), o)
    return bool(ok), list(o)


@pytest.mark.parametrize("nu,nrest,npol", [(32, 64, 2), (64, 64, 2), (64, 8, 4)])
def test_buckets_follow_the_windows(L, nu, nrest, npol):
    n = {w: _layout(L, nu, nu, nrest, npol, w)[1][1] for w in (1, 12, 38, 100, 300, 600, 2000, 100000)}
    assert n[1] == n[12] == n[38] == 32
    for w in (100, 300, 600):
        assert 1 <= n[w] <= 2 * 8 * 152 // w, (w, n[w])
    assert n[2000] == n[100000] <= max(1, nu * nu // 2048)


def test_layout_limits(L):
    lim = (C.c_int * 2)()
    L.limits(lim)
    rng = random.Random(1)
    for _ in range(3000):
        nu, nv = (2 * round(10 ** rng.uniform(0.0, 4.2)) for _ in range(2))
        nrest, npol, w = round(10 ** rng.uniform(0.0, 3.5)), rng.randint(1, 4), round(10 ** rng.uniform(0.0, 5.0))
        ok, (S, nst, ushift, nuk) = _layout(L, nu, nv, nrest, npol, w)
        assert ok
        assert 1 <= S <= nv and nst * S >= nv > (nst - 1) * S and nst <= lim[1]
        assert nuk == (nu + (1 << ushift) - 1) >> ushift and S * nuk <= lim[0]
