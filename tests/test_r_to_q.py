"""chi0(R, tau) -> chi0(q, i omega) against the same two sums on the host, for meshes of every kernel size: cells that
are their own inverse only, pairs only beside the home cell, both, odd and even meshes."""
import numpy as np
import pytest

from paper_2407_19930_gb300 import librpa_gpu as L
from paper_2407_19930_gb300 import synthetic as syn
from oracle import grid as ogrid

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kmesh", [(1, 1, 1), (2, 2, 2), (3, 3, 1), (4, 4, 1), (5, 4, 1), (4, 2, 4), (7, 5, 1)])
def test_r_to_q(kmesh):
    inp = syn.make_inputs(syn.cubic_two_atom(nao=3, naux=5, nlow=1, kmesh=kmesh), 51, vscale=1e-3)
    grid = ogrid.make_grid(6, *inp.delta_range)
    st, nw = inp.st, len(grid["omega"])
    o = L.librpa_gpu_default_opts()
    h = L.librpa_gpu_create(o)
    try:
        L.set_inputs(h, inp, grid)
        chi = L.librpa_gpu_chi0(h, out=(st.nk, nw, st.naux))
        tau = np.array([[L.librpa_gpu_get_chi0_tau(h, j, r, st.naux) for r in range(st.nk)] for j in range(nw)])
    finally:
        L.librpa_gpu_destroy(h)
    cells, n = syn.bvk_cells(kmesh), np.array(kmesh)   # (the q of the mesh have the same indices)
    phase = np.exp(2j * np.pi * ((cells[:, None] * cells[None]) % n / n).sum(-1))
    ref = np.einsum("kj,qr,jrmn->qkmn", grid["gamma"], phase, tau)
    # a rounding per term of the two sums
    bound = 2.0 ** -52 * (st.nk + nw) * np.einsum("kj,jrmn->kmn", np.abs(grid["gamma"]), np.abs(tau)).max(axis=(1, 2))
    assert (np.abs(chi - ref).max(axis=(2, 3)) <= bound[None]).all()
