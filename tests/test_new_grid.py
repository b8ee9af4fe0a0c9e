"""A handle whose grid changes gives what a fresh handle gives, also when the number of points takes the FP64 contraction
from the FP64 pipes to digit planes or back."""
import numpy as np
import pytest

from paper_2407_19930_gb300 import librpa_gpu as L
from paper_2407_19930_gb300 import synthetic as syn
from oracle import grid as ogrid

pytestmark = pytest.mark.gpu


def _chi(h, inp, ntau):
    L.librpa_gpu_chi0(h)
    planes = L.librpa_gpu_get_stats(h)["flop_exec_gemm_chi0"] > 0
    tau = np.array([[L.librpa_gpu_get_chi0_tau(h, t, r, inp.st.naux) for r in range(inp.st.nk)] for t in range(ntau)])
    return planes, tau


def test_grid_of_another_size():
    # 2.6e8 contraction flops a time point: one on either side of 5e8
    st = syn.Structure(lat=np.eye(3) * 6.5, pos=np.array([[0.0, 0.0, 0.0], [3.1, 0.4, 0.2], [0.3, 3.0, 2.2]]),
                       n_ao=np.array([16, 16, 3]), n_aux=np.array([64, 33, 1]), n_low=np.array([2, 2, 1]), kmesh=(3, 1, 1))
    inp = syn.make_inputs(st, 91, vscale=3e-4)
    grids = {n: ogrid.make_grid(n, *inp.delta_range) for n in (1, 6)}
    fresh = {}
    for n, g in grids.items():
        h = L.librpa_gpu_create(L.librpa_gpu_default_opts())
        try:
            L.set_inputs(h, inp, g)
            fresh[n] = _chi(h, inp, n)
        finally:
            L.librpa_gpu_destroy(h)
    assert not fresh[1][0] and fresh[6][0]
    h = L.librpa_gpu_create(L.librpa_gpu_default_opts())
    try:
        L.set_inputs(h, inp, grids[1])
        for n in (1, 6, 1):
            g = grids[n]
            L.librpa_gpu_set_grid(h, g["tau"], g["omega"], g["w_omega"], g["gamma"])
            planes, tau = _chi(h, inp, n)
            assert planes == fresh[n][0] and np.array_equal(tau, fresh[n][1])
    finally:
        L.librpa_gpu_destroy(h)
