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


@pytest.mark.parametrize("spread", [4, 16, 30])
def test_atomic_orbitals(spread):
    inp, grid = _inputs()
    st = inp.st
    ec, ec_q, _ = _run(inp, grid)
    e = np.random.default_rng(6).integers(-spread // 2, spread // 2 + 1, st.nao)
    a = 2.0 ** e
    off = np.concatenate([[0], np.cumsum(st.n_ao)])
    s = copy.copy(inp)
    s.wfc = inp.wfc * a
    s.lri = [(I, K, R, C / a[off[I]:off[I + 1], None] / a[off[K]:off[K + 1]]) for I, K, R, C in inp.lri]
    ec2, ec_q2, _ = _run(s, grid)
    # products of 63-bit operands whose rows spread over at most 2^6 more than without the rescaling (2^-57 of
    # an element), each stored with 53 bits: the two energies differ by a few times 2^-53 of the sums over N_aux
    assert abs(ec2 - ec) <= 1e-12 * abs(ec) and np.abs(ec_q2 - ec_q).max() <= 1e-12 * np.abs(ec_q).max()


def test_green_function_in_the_callers_orbitals():
    inp, grid = _inputs()
    st = inp.st
    a = 2.0 ** np.random.default_rng(6).integers(-15, 16, st.nao)
    s = copy.copy(inp)
    s.wfc = inp.wfc * a
    s.lri = [(I, K, R, np.zeros_like(C)) for I, K, R, C in inp.lri]
    g = []
    for x in (inp, s):
        h = L.librpa_gpu_create(L.librpa_gpu_default_opts())
        try:
            L.set_inputs(h, x, grid)
            L.librpa_gpu_chi0(h)
            g.append([L.librpa_gpu_get_green(h, it, r, st.nao) for it in range(len(grid["tau"])) for r in range(st.nk)])
        finally:
            L.librpa_gpu_destroy(h)
    assert np.array_equal(np.array(g[1]), np.array(g[0]) * a[:, None] * a)   # powers of two
