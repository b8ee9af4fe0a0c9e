"""The FP64 mode does not depend on the norms of the basis functions: E_c and its parts are the same when auxiliary
functions or NAOs are rescaled by powers of two, also far beyond the bits that a digit plane holds below its row's
largest element."""
import copy

import numpy as np
import pytest

from paper_2407_19930_gb300 import librpa_gpu as L
from paper_2407_19930_gb300 import synthetic as syn
from oracle import grid as ogrid, pipeline

pytestmark = pytest.mark.gpu


def _inputs():
    # N_aux 98 (8 planes in the ln det) and 1.6e9 contraction flops (8 planes there); a real q and a complex pair
    st = syn.Structure(lat=np.eye(3) * 6.5, pos=np.array([[0.0, 0.0, 0.0], [3.1, 0.4, 0.2], [0.3, 3.0, 2.2]]),
                       n_ao=np.array([16, 16, 3]), n_aux=np.array([64, 33, 1]), n_low=np.array([2, 2, 1]), kmesh=(3, 1, 1))
    inp = syn.make_inputs(st, 91, vscale=3e-4)
    return inp, ogrid.make_grid(6, *inp.delta_range)


def _run(inp, grid):
    h = L.librpa_gpu_create(L.librpa_gpu_default_opts())
    try:
        L.set_inputs(h, inp, grid)
        L.librpa_gpu_chi0(h)
        return L.librpa_gpu_ec(h, inp.st.nk, len(grid["omega"]))
    finally:
        L.librpa_gpu_destroy(h)


@pytest.mark.parametrize("spread", [10, 24, 40])
def test_auxiliary_functions(spread):
    inp, grid = _inputs()
    st = inp.st
    ec, ec_q, ec_w = _run(inp, grid)
    assert abs(ec - pipeline.rpa_energy(inp, grid)["ec"]) < 1e-8
    d = 2.0 ** np.random.default_rng(5).integers(-spread // 2, spread // 2 + 1, st.naux)
    off = np.concatenate([[0], np.cumsum(st.n_aux)])
    s = copy.copy(inp)
    s.lri = [(I, K, R, C / d[off[I]:off[I + 1], None, None]) for I, K, R, C in inp.lri]
    s.vq = inp.vq * d[:, None] * d[None, :]
    ec2, ec_q2, ec_w2 = _run(s, grid)
    # powers of two change no rounding
    assert ec2 == ec and np.array_equal(ec_q2, ec_q) and np.array_equal(ec_w2, ec_w)
