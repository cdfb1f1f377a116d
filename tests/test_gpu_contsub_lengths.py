"""Continuum subtraction over cells of lengths around the steps of the count
reads (16 bytes a lane where a cell's entries are whole quadruples), against the
oracle's fit on the same cube, with a line-free mask and with a fit set of a few
channels; entries without a contribution, and whole cells, give zeros."""
import numpy as np
import pytest

from tests.test_gpu_contsub import V, _kernel_check, _line_free, _stack  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("planes,nrest", [(1, 31), (1, 32), (2, 511), (2, 512), (1, 1025), (4, 257), (2, 2050)])
@pytest.mark.parametrize("order", [0, 1, 3])
def test_lengths_against_oracle_fit(V, planes, nrest, order):  # noqa: F811
    from paper_2609_01897_gb300 import synth
    pols = {1: (1,), 2: (2,), 4: (4,)}[planes]
    wl = synth.random_case(5 + planes, "cuda", nsrc=6, max_rows=150, npol_choices=pols, nrest=nrest)
    wl.npol = planes
    few = np.zeros(nrest, dtype=bool)
    few[np.linspace(nrest // 8, nrest - nrest // 8, 6).astype(int)] = True
    st = _stack(V, wl, V.PREC_MIXED)
    try:
        cube = st.read_cube(device=True, f64=True)
        wv = (cube["sum_wv"][..., 0] + 1j * cube["sum_wv"][..., 1]).cpu().numpy()
        w = cube["sum_w"].cpu().numpy()
        assert (w > 0).sum() > 100 and (w.reshape(-1, w.shape[-1]) == 0).any()
        for free in (_line_free(nrest, order), few):
            got = st.contsub(free, order).cpu().numpy()
            _kernel_check(got, wv, w, free, order)
            assert not got[w == 0].any()
    finally:
        st.close()
