"""Digit-plane kernels at the edges of their tiles: numbers of functions per atom next to the widths the kernels
are built for (16 functions an atom in the O assembly, 32 / 48 / 64 columns a GEMM tile, panels of 64), one function
an atom, and every plane count of the ln det, against the CPU oracle."""
import functools

import numpy as np
import pytest

from paper_2407_19930_gb300 import librpa_gpu as L
from paper_2407_19930_gb300 import synthetic as syn
from oracle import grid as ogrid, pipeline

pytestmark = pytest.mark.gpu

# (functions, auxiliary functions, occupied bands) per atom, mesh
SHAPES = {
    "largest_atom": ([(16, 64, 2), (16, 33, 2), (3, 1, 1)], (3, 1, 1)),       # N_aux 98: panels 64 + 34
    "beyond_largest_atom": ([(17, 48, 2), (5, 48, 1)], (2, 1, 1)),            # N_aux 96: the line of the 8-plane ln det
    "below_line": ([(9, 47, 2), (5, 48, 1)], (2, 1, 1)),                      # N_aux 95: the FP64 pipes
    "smallest_atom": ([(1, 31, 1), (2, 65, 1), (13, 33, 2)], (3, 1, 1)),      # N_aux 129: a panel of one row
}
POS = [[0.0, 0.0, 0.0], [3.1, 0.4, 0.2], [0.3, 3.0, 2.2]]


@functools.lru_cache(maxsize=None)
def _reference(name):
    species, kmesh = SHAPES[name]
    n = [np.array(x) for x in zip(*species)]
    st = syn.Structure(lat=np.eye(3) * 6.5, pos=np.array(POS[:len(species)]), n_ao=n[0], n_aux=n[1], n_low=n[2],
                       kmesh=kmesh)
    inp = syn.make_inputs(st, 91, vscale=3e-4)
    grid = ogrid.make_grid(6, *inp.delta_range)
    return inp, grid, pipeline.rpa_energy(inp, grid)


def _energy(inp, grid, precision, ec_slices=0):
    o = L.librpa_gpu_default_opts()
    o.precision, o.ec_slices = precision, ec_slices
    h = L.librpa_gpu_create(o)
    try:
        L.set_inputs(h, inp, grid)
        L.librpa_gpu_chi0(h)
        st = inp.st
        tau = np.array([[L.librpa_gpu_get_chi0_tau(h, it, iR, st.naux) for iR in range(st.nk)]
                        for it in range(len(grid["tau"]))])
        return tau, L.librpa_gpu_ec(h, st.nk, len(grid["omega"]))
    finally:
        L.librpa_gpu_destroy(h)


@pytest.mark.parametrize("precision", [L.LIBRPA_FP64, L.LIBRPA_FP64_TC])
@pytest.mark.parametrize("name", list(SHAPES))
def test_tile_edges(name, precision):
    """chi0(R, tau) to 1e-10 of its largest element (39 bits per operand: 2^-39 times the ~50 digit products that add
    up at random), E_c to 1e-8 Ha: the tolerances of the element-wise parity tests."""
    inp, grid, ref = _reference(name)
    tau, (ec, ec_q, _) = _energy(inp, grid, precision)
    assert np.abs(tau - ref["chi_tau"]).max() < 1e-10 * np.abs(ref["chi_tau"]).max()
    assert abs(ec - ref["ec"]) < 1e-8
    assert np.abs(ec_q - ref["ec_q"]).max() < 1e-8


@pytest.mark.parametrize("slices", [1, 2, 3, 4, 5])
def test_lndet_planes(slices):
    """ln det with every plane count on a real q and a complex pair.  Elements of an operand are rounded by at most
    2^(-8 S) of their row's largest, so an element of L^H chi0 L is off by at most 2 N_aux 2^(-8 S) of its row's scale
    per product and E_c (second order in it) by a few times that."""
    inp, grid, ref = _reference("smallest_atom")
    _, (ec, ec_q, _) = _energy(inp, grid, L.LIBRPA_FP64_TC, slices)
    tol = 8.0 * inp.st.naux * 2.0 ** (-8 * slices) * np.abs(ref["ec_q"]).max() + 1e-10
    assert np.isfinite(ec)
    assert np.abs(ec_q - ref["ec_q"]).max() < tol
