"""A bounded wait that runs out in any handle of a merged batch fails the batch (it left that handle's result
unfinished); the next run gives every handle's own energy."""
import pytest

from paper_2407_19930_gb300 import librpa_gpu as L
from paper_2407_19930_gb300 import synthetic as syn
from oracle import grid as ogrid, pipeline

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [L.LIBRPA_FP64, L.LIBRPA_FP64_TC])
@pytest.mark.parametrize("late", [1, 2])
def test_wait_runs_out_in_a_later_handle(precision, late):
    inp = syn.config_cubic()
    grid = ogrid.make_grid(6, *inp.delta_range)
    hs, b = [], None
    try:
        for i in range(3):
            o = L.librpa_gpu_default_opts()
            o.precision = precision
            o.test_stall_gemms = L.LIBRPA_TEST_STALL_OASM if i == late else 0
            hs.append(L.librpa_gpu_create(o))
            L.set_inputs(hs[-1], inp, grid)
        b = L.librpa_gpu_batch_create(hs)
        with pytest.raises(L.LibrpaError) as e:
            L.librpa_gpu_batch_run(b)
        assert e.value.code == L.LIBRPA_E_TIMEOUT
        ec = L.librpa_gpu_batch_run(b)
    finally:
        L.librpa_gpu_batch_destroy(b)
        for h in hs:
            L.librpa_gpu_destroy(h)
    ref = pipeline.rpa_energy(inp, grid)["ec"]
    assert max(abs(e - ref) for e in ec) < 1e-8
