"""The bounded-wait failure paths of the 8-plane GEMM and of the tensor-core O assembly, made to run without a GPU
fault (see test_timeout): the call reports LIBRPA_E_TIMEOUT, the handle's next calls give the oracle's energy."""
import functools

import numpy as np
import pytest

from paper_2407_19930_gb300 import librpa_gpu as L
from paper_2407_19930_gb300 import synthetic as syn
from oracle import grid as ogrid, pipeline

pytestmark = pytest.mark.gpu
W, A = L.LIBRPA_TEST_STALL_WIDE, L.LIBRPA_TEST_STALL_OASM


@functools.lru_cache(maxsize=None)
def _reference(name):
    # "panels": N_aux 98, two panels in the ln det, whose real matrices (one k point) take 8-plane panel products
    inp = syn.config_cubic() if name == "cubic" else syn.make_inputs(
        syn.Structure(lat=np.eye(3) * 6.5, pos=np.array([[0.0, 0.0, 0.0], [3.1, 0.4, 0.2]]), n_ao=np.array([6, 5]),
                      n_aux=np.array([60, 38]), n_low=np.array([2, 1]), kmesh=(1, 1, 1)), 91, vscale=3e-4)
    grid = ogrid.make_grid(6, *inp.delta_range)
    return inp, grid, pipeline.rpa_energy(inp, grid)["ec"]


@pytest.mark.parametrize("name,precision,stall,stage", [
    ("cubic", L.LIBRPA_FP64, W, "chi0"),
    ("cubic", L.LIBRPA_FP64, 3 * W, "chi0"),
    ("cubic", L.LIBRPA_FP64, A, "chi0"),
    ("cubic", L.LIBRPA_FP64_TC, A, "chi0"),
    ("cubic", L.LIBRPA_SPLIT, A, "chi0"),
    ("panels", L.LIBRPA_FP64, W, "ec"),
    ("panels", L.LIBRPA_FP64_TC, W, "ec"),
])
def test_wait_runs_out_then_the_handle_recovers(name, precision, stall, stage):
    inp, grid, ref = _reference(name)
    o = L.librpa_gpu_default_opts()
    o.precision, o.test_stall_gemms = precision, stall
    h = L.librpa_gpu_create(o)
    try:
        L.set_inputs(h, inp, grid)
        if stage == "ec":
            L.librpa_gpu_chi0(h)
        with pytest.raises(L.LibrpaError) as e:
            L.librpa_gpu_chi0(h) if stage == "chi0" else L.librpa_gpu_ec(h)
        assert e.value.code == L.LIBRPA_E_TIMEOUT
        if stage == "chi0":
            L.librpa_gpu_chi0(h)
        ec, _, _ = L.librpa_gpu_ec(h)
    finally:
        L.librpa_gpu_destroy(h)
    # the element-wise tests' bound; 0.1 meV per atom in the mixed mode
    assert abs(ec - ref) < (1e-8 if precision != L.LIBRPA_SPLIT else 1e-4 / 27.2 * inp.st.natoms)
