"""The single-launch form (grid -4) gives up at once when a wait runs out: its CTAs wait
for their copies in flight, which take microseconds, and for nothing else."""
import time

import pytest

pytestmark = pytest.mark.gpu


def test_gives_up_without_delay_and_the_next_call_is_exact():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_1611_04959_gb300 as daq
    F, C, X, N = 1, 24, 54, 280_000
    g = torch.Generator(device="cuda").manual_seed(4)
    x = torch.randint(1790, 1811, (F, C, X, N), generator=g, device="cuda", dtype=torch.int16)
    ref = daq.process_fills(x, grid=200, threshold=150)
    gave_up = 0
    for k in range(6):
        torch.cuda.synchronize()
        t0 = time.monotonic()
        # 1 ns: the scanner's wait for a record, or the count role's for the compact role, runs out at once
        r = daq.process_fills(x, grid=-4, lag_tiles=640 + 100 * k, wait_limit_ns=1, threshold=150, allow=(daq.DAQ_ETIMEOUT,))
        took = time.monotonic() - t0
        assert r["status"] in (daq.DAQ_OK, daq.DAQ_ETIMEOUT)
        gave_up += r["status"] == daq.DAQ_ETIMEOUT
        assert took < 1.0
    assert gave_up
    a = daq.process_fills(x, grid=-4, threshold=150)
    assert a["status"] == daq.DAQ_OK and list(a["counts"]) == list(ref["counts"])
    n, m = a["n_rows"], a["n_islands"]
    assert torch.equal(a["outputs"].hdr[: 3 * m], ref["outputs"].hdr[: 3 * m])
    assert torch.equal(a["outputs"].pool[:n], ref["outputs"].pool[:n]) and torch.equal(a["q"], ref["q"])
