"""NaN in an input reaches every result it enters, in each arithmetic of the contraction, and no other."""
import numpy as np
import pytest

from paper_2407_19930_gb300 import librpa_gpu as L
from paper_2407_19930_gb300 import synthetic as syn
from oracle import grid as ogrid, pipeline

pytestmark = pytest.mark.gpu


def _inputs():
    # 1.6e9 contraction flops: 8 planes in the FP64 mode
    st = syn.Structure(lat=np.eye(3) * 6.5, pos=np.array([[0.0, 0.0, 0.0], [3.1, 0.4, 0.2], [0.3, 3.0, 2.2]]),
                       n_ao=np.array([16, 16, 3]), n_aux=np.array([64, 33, 1]), n_low=np.array([2, 2, 1]), kmesh=(3, 1, 1))
    inp = syn.make_inputs(st, 91, vscale=3e-4)
    return inp, ogrid.make_grid(6, *inp.delta_range)


@pytest.mark.parametrize("value", [np.nan, np.inf])
@pytest.mark.parametrize("precision", [L.LIBRPA_FP64, L.LIBRPA_FP64_TC, L.LIBRPA_SPLIT])
def test_coefficient(precision, value):
    inp, grid = _inputs()
    st, mu = inp.st, 64 + 7   # function 7 of atom 1
    ref = pipeline.rpa_energy(inp, grid)["chi_tau"]
    for x, (I, K, R, C) in enumerate(inp.lri):
        if I == 1 and K == 1 and tuple(R) == (0, 0, 0):
            C = C.copy()
            C[7, 3, 5] = value
            inp.lri[x] = (I, K, R, C)
    o = L.librpa_gpu_default_opts()
    o.precision = precision
    h = L.librpa_gpu_create(o)
    try:
        L.set_inputs(h, inp, grid)
        L.librpa_gpu_chi0(h)
        tau = np.array([[L.librpa_gpu_get_chi0_tau(h, t, r, st.naux) for r in range(st.nk)] for t in range(6)])
        with pytest.raises(L.LibrpaError) as e:
            L.librpa_gpu_ec(h)
        assert e.value.code == L.LIBRPA_E_NOT_PD
    finally:
        L.librpa_gpu_destroy(h)
    bad = np.zeros((st.naux, st.naux), bool)
    bad[mu, :] = bad[:, mu] = True
    assert not np.isfinite(tau[..., bad]).any()
    tol = {L.LIBRPA_FP64: 1e-10, L.LIBRPA_FP64_TC: 1e-10, L.LIBRPA_SPLIT: 1e-5}[precision]   # as without the NaN
    assert np.abs(tau - ref)[..., ~bad].max() < tol * np.abs(ref).max()


@pytest.mark.parametrize("precision", [L.LIBRPA_FP64, L.LIBRPA_FP64_TC])
def test_orbitals_without_a_number(precision):
    """Kohn-Sham coefficients that are all NaN give results that are NaN, not an error of the imaginary part."""
    inp, grid = _inputs()
    inp.wfc = np.full_like(inp.wfc, np.nan)
    o = L.librpa_gpu_default_opts()
    o.precision = precision
    h = L.librpa_gpu_create(o)
    try:
        L.set_inputs(h, inp, grid)
        L.librpa_gpu_chi0(h)
        assert np.isnan(L.librpa_gpu_get_chi0_tau(h, 0, 0, inp.st.naux)).all()
    finally:
        L.librpa_gpu_destroy(h)
