"""Requests that fit the routes of least memory (FP64 mode: the FP64 pipes; the others: the O assembly without digit
planes of its operands) run within that much memory, and batches bound their workspaces together."""
import functools

import numpy as np
import pytest

from paper_2407_19930_gb300 import librpa_gpu as L
from paper_2407_19930_gb300 import synthetic as syn
from oracle import grid as ogrid

pytestmark = pytest.mark.gpu
NTAU = 8


@functools.lru_cache(maxsize=None)
def _inputs():
    inp = syn.make_inputs(syn.random_cell(np.random.default_rng(12), 12, (1, 1, 1)), 12, vscale=2e-4)
    return inp, ogrid.make_grid(NTAU, *inp.delta_range)


def _pipes_bytes(st):
    """Device bytes of an FP64 request on the FP64 pipes: inputs, G, chi0(R, tau), chi0(q, i omega), packed C (and the
    gathers, N, X and O of a batch of points, at most 2^27 doubles), L(q), W and A; 2% for tables and alignment."""
    n2, a2, nk = st.naux ** 2, st.nao ** 2, st.nk
    lri = 8 * 60 * 13 * 13 * 100 * st.natoms   # at most 100 neighbours an atom
    return int(1.02 * (16 * nk * (a2 + n2) + 16 * NTAU * nk * a2 + 24 * NTAU * nk * n2 + lri + 8 * 2 ** 27 +
                       16 * n2 * (nk + 2 * NTAU)))


def _run(inp, grid, precision, budget=0):
    o = L.librpa_gpu_default_opts()
    o.precision, o.hbm_budget = precision, budget
    h = L.librpa_gpu_create(o)
    try:
        L.set_inputs(h, inp, grid)
        L.librpa_gpu_chi0(h)
        peak = L.librpa_gpu_get_stats(h)["bytes_device_peak"]
        ec = [L.librpa_gpu_ec(h, inp.st.nk, NTAU)[0]]
        L.librpa_gpu_chi0(h)   # a second pass within the same budget
        ec.append(L.librpa_gpu_ec(h, inp.st.nk, NTAU)[0])
        return ec, peak, L.librpa_gpu_get_stats(h)
    finally:
        L.librpa_gpu_destroy(h)


def test_fp64_within_the_pipes_memory():
    inp, grid = _inputs()
    ec, peak_chi0, st = _run(inp, grid, L.LIBRPA_FP64)
    peak, pipes = st["bytes_device_peak"], _pipes_bytes(inp.st)
    assert pipes < peak
    # the ln det alone falls back, then the contraction (beside whose smaller workspace the ln det's planes may fit)
    for budget in ((peak_chi0 + peak) // 2, pipes):
        e, _, s = _run(inp, grid, L.LIBRPA_FP64, budget)
        assert s["bytes_device_peak"] <= budget
        assert max(abs(x - ec[0]) for x in e) < 1e-8
    assert s["flop_exec_gemm_chi0"] == 0


@pytest.mark.parametrize("precision,budget", [(L.LIBRPA_FP64, 3.95e9), (L.LIBRPA_FP64_TC, 7.95e9), (L.LIBRPA_SPLIT, 7.2e9)])
def test_slab_within_the_least_memory(precision, budget):
    """Graphene slab and molecule, one k point, 8 points: 3.83, 7.86 and 7.10 GB without the digit planes of the FP64
    mode and of the O assembly's operands."""
    inp = syn.config_graphene(kmesh=(1, 1, 1))
    grid = ogrid.make_grid(NTAU, *inp.delta_range)
    ec, _, s0 = _run(inp, grid, precision)
    assert s0["bytes_device_peak"] > budget
    e, _, s = _run(inp, grid, precision, int(budget))
    assert s["bytes_device_peak"] <= budget
    tol = 1e-8 if precision != L.LIBRPA_SPLIT else 1e-4 / 27.2 * inp.st.natoms
    assert max(abs(x - ec[0]) for x in e) < tol


def test_fp64_batch_bounds_its_workspaces():
    """20 structures whose workspaces would each take about 1 GiB or more: at most 16 GiB together, beside what the handles
    keep (below 0.15 GB each)."""
    import torch
    inp = syn.config_mixed()
    grid = ogrid.make_grid(10, *inp.delta_range)
    hs, b = [], None
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    try:
        for _ in range(20):
            hs.append(L.librpa_gpu_create(L.librpa_gpu_default_opts()))
            L.set_inputs(hs[-1], inp, grid)
        b = L.librpa_gpu_batch_create(hs)
        ec = L.librpa_gpu_batch_run(b)
        used = free - torch.cuda.mem_get_info()[0]
    finally:
        L.librpa_gpu_batch_destroy(b)
        for h in hs:
            L.librpa_gpu_destroy(h)
    assert np.ptp(ec) <= 1e-12 * abs(ec[0])
    assert used < (16 << 30) + 20 * 0.15e9


def test_server_admits_what_fits_without_planes():
    inp, grid = _inputs()
    o = L.librpa_gpu_default_opts()
    h = L.librpa_gpu_create(o)
    try:
        L.set_inputs(h, inp, grid)
        budget = int(L.librpa_gpu_estimate_bytes(h)) - (64 << 20)
        L.librpa_gpu_chi0(h)
        ec = L.librpa_gpu_ec(h)[0]
    finally:
        L.librpa_gpu_destroy(h)
    s = L.librpa_gpu_server_create(slots=1, hbm_budget=budget)
    r = None
    try:
        r = L.librpa_gpu_server_request(s, o)
        L.set_inputs(r, inp, grid)
        res = L.librpa_gpu_server_wait(s, L.librpa_gpu_server_submit(s, r), 120.0)
        assert res["status"] == L.LIBRPA_OK and abs(res["ec"] - ec) < 1e-8
        assert res["bytes_peak"] <= res["bytes_reserved"] <= budget
    finally:
        L.librpa_gpu_server_destroy(s)
        if r:
            L.librpa_gpu_destroy(r)
