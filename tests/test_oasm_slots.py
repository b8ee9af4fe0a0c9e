"""O assembly with many auxiliary functions per atom and tiles whose warps mostly have no row (they run ahead of the
others through the accumulator slots): every pass gives the same bits, and the oracle's chi0."""
import numpy as np
import pytest

from paper_2407_19930_gb300 import librpa_gpu as L
from paper_2407_19930_gb300 import synthetic as syn
from oracle import grid as ogrid, pipeline

pytestmark = pytest.mark.gpu


# slots of 5, 3 and 8 planes: 3, 5 and 2; bounds: those of the element-wise tests, 2^-17 for 23-bit operands
@pytest.mark.parametrize("precision,tol", [(L.LIBRPA_FP64_TC, 1e-10), (L.LIBRPA_SPLIT, 2.0 ** -17), (L.LIBRPA_FP64, 1e-10)])
def test_passes_agree(precision, tol):
    st = syn.Structure(lat=np.eye(3) * 6.5, pos=np.array([[0.0, 0.0, 0.0], [3.1, 0.4, 0.2]]), n_ao=np.array([4, 3]),
                       n_aux=np.array([211, 128]), n_low=np.array([1, 1]), kmesh=(3, 3, 2))
    inp = syn.make_inputs(st, 17, vscale=1e-4)
    grid = ogrid.make_grid(8, *inp.delta_range)
    ref = pipeline.rpa_energy(inp, grid)["chi_tau"]
    o = L.librpa_gpu_default_opts()
    o.precision = precision
    h = L.librpa_gpu_create(o)
    try:
        L.set_inputs(h, inp, grid)
        got = []
        for _ in range(10):
            L.librpa_gpu_chi0(h)
            got.append(np.array([L.librpa_gpu_get_chi0_tau(h, t, r, st.naux) for t in range(8) for r in range(0, st.nk, 5)]))
        assert L.librpa_gpu_get_stats(h)["flop_exec_gemm_chi0"] > 0
    finally:
        L.librpa_gpu_destroy(h)
    assert all(np.array_equal(g, got[0]) for g in got)
    ref = np.array([ref[t][r] for t in range(8) for r in range(0, st.nk, 5)])
    assert np.abs(got[0] - ref).max() < tol * np.abs(ref).max()
