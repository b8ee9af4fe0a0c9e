"""FP64 requests on 8 digit planes over the forms that the kernels take them in, against the CPU oracle: atoms with more
NAOs than the tensor-core O assembly holds, one function per atom, neighbour lists of every gather kernel."""
import numpy as np
import pytest

from paper_2407_19930_gb300 import librpa_gpu as L
from paper_2407_19930_gb300 import synthetic as syn
from oracle import grid as ogrid, pipeline

pytestmark = pytest.mark.gpu

POS3 = [[0.0, 0.0, 0.0], [3.1, 0.4, 0.2], [0.3, 3.0, 2.2]]
# lattice constant, positions, (NAO, auxiliary functions, occupied bands) per atom, mesh; all above 5e8 contraction flops
SHAPES = {
    "more_naos_than_the_o_assembly": (6.5, POS3[:2], [(17, 48, 2), (16, 48, 2)], (3, 2, 1)),
    "one_function_atoms": (6.5, POS3, [(1, 31, 1), (16, 65, 2), (13, 33, 2)], (3, 1, 1)),
    "columns_256": (2.9, POS3[:1], [(7, 24, 1)], (2, 2, 1)),       # 33 neighbours: K 231
    "columns_512": (2.9, POS3[:1], [(9, 16, 1)], (2, 2, 1)),       # K 297
    "columns_beyond": (2.9, POS3[:1], [(16, 9, 2)], (2, 1, 1)),    # K 528
}


@pytest.mark.parametrize("name", list(SHAPES))
def test_fp64(name):
    a, pos, species, kmesh = SHAPES[name]
    n = [np.array(x) for x in zip(*species)]
    inp = syn.make_inputs(syn.Structure(lat=np.eye(3) * a, pos=np.array(pos), n_ao=n[0], n_aux=n[1], n_low=n[2], kmesh=kmesh),
                          92, vscale=3e-4)
    grid = ogrid.make_grid(6, *inp.delta_range)
    ref = pipeline.rpa_energy(inp, grid)
    h = L.librpa_gpu_create(L.librpa_gpu_default_opts())
    try:
        L.set_inputs(h, inp, grid)
        L.librpa_gpu_chi0(h)
        assert L.librpa_gpu_get_stats(h)["flop_exec_gemm_chi0"] > 0   # on digit planes
        st = inp.st
        tau = np.array([[L.librpa_gpu_get_chi0_tau(h, it, r, st.naux) for r in range(st.nk)] for it in range(6)])
        ec, ec_q, _ = L.librpa_gpu_ec(h, st.nk, 6)
    finally:
        L.librpa_gpu_destroy(h)
    # the element-wise tests' bounds of FP64
    assert np.abs(tau - ref["chi_tau"]).max() < 1e-10 * np.abs(ref["chi_tau"]).max()
    assert abs(ec - ref["ec"]) < 1e-8 and np.abs(ec_q - ref["ec_q"]).max() < 1e-8


@pytest.mark.parametrize("slices", [1, 2, 3, 4, 5])
def test_planes_of_the_lndet(slices):
    """Elements are cut to 2^(-8 S) of their row's largest; N_aux = 129 of them, off either way, add up to about 2^3.5 times
    that, so E_c is off by less than 2^4 2^(-8 S) of itself (one plane: a sixteenth), beside the rounding of the sums."""
    a, pos, species, kmesh = SHAPES["one_function_atoms"]
    n = [np.array(x) for x in zip(*species)]
    inp = syn.make_inputs(syn.Structure(lat=np.eye(3) * a, pos=np.array(pos), n_ao=n[0], n_aux=n[1], n_low=n[2], kmesh=kmesh),
                          92, vscale=3e-4)
    grid = ogrid.make_grid(6, *inp.delta_range)
    ref = pipeline.rpa_energy(inp, grid)["ec"]
    o = L.librpa_gpu_default_opts()
    o.ec_slices = slices
    h = L.librpa_gpu_create(o)
    try:
        L.set_inputs(h, inp, grid)
        L.librpa_gpu_chi0(h)
        ec = L.librpa_gpu_ec(h)[0]
    finally:
        L.librpa_gpu_destroy(h)
    assert abs(ec - ref) < 2.0 ** (4 - 8 * slices) * abs(ref) + 1e-11
