"""The phased form's way out: a chunk's aggregates that never come make the call give up
after the caller's limit, with DAQ_ETIMEOUT, and the next call is exact.

The aggregates are made to go missing from outside: while the kernel runs, copies on
another stream clear the words that its CTAs publish (a cleared word reads as one that
is not there yet), which a correct program never does."""
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_1611_04959_gb300 as daq
    return dict(torch=torch, daq=daq)


# 1.2 s: the wait for the aggregates runs out first.  4.7 s: no wait of a CTA on its own
# warps, which depend on that one, may end it sooner (theirs without other CTAs is 4 s).
@pytest.mark.parametrize("limit", [1.2, 4.7])
def test_gives_up_at_the_limit_and_the_next_call_is_exact(env, limit):
    torch, daq = env["torch"], env["daq"]
    F, C, X, N = 1, 24, 54, 280_000
    g = torch.Generator(device="cuda").manual_seed(3)
    x = torch.randint(1790, 1811, (F, C, X, N), generator=g, device="cuda", dtype=torch.int16)
    tiles = C * -(-N // 448)
    assert tiles >= 14 * torch.cuda.get_device_properties(0).multi_processor_count  # phased
    out = daq.Outputs(torch, "cuda", F, C, X, C * N // 2, C * N)
    ws = torch.zeros(daq.daq_workspace_size(C, X, N, F, daq.make_params()), dtype=torch.uint8, device="cuda")

    def up(v):
        return -(-v // 256) * 256

    words = up(up(up(512 + 8 * (F + 1)) + 4 * F) + 4 * F * C)    # where the tiles' words lie
    zeros = torch.zeros(4 * tiles, dtype=torch.uint8, pin_memory=True)
    main, side = torch.cuda.current_stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    torch.cuda._sleep(4_000_000)                                # about 2 ms: the copies are under way by then
    t0 = time.monotonic()
    daq.process_fills(x, outputs=out, workspace=ws, sync=False, wait_limit_ns=int(limit * 1e9))
    with torch.cuda.stream(side):
        for _ in range(1500):
            ws[words: words + 4 * tiles].copy_(zeros, non_blocking=True)
    counts = np.zeros(4, np.int64)
    rc = daq.daq_read_counts(out.counts.data_ptr(), counts, main)
    took = time.monotonic() - t0
    torch.cuda.synchronize()
    assert rc == daq.DAQ_ETIMEOUT and counts[2] & daq.DAQ_DEV_TIMEOUT
    assert limit * 0.98 < took < limit + 1.0

    a = daq.process_fills(x, outputs=out, workspace=ws)
    b = daq.process_fills(x, grid=200)
    assert a["status"] == b["status"] == daq.DAQ_OK and list(a["counts"]) == list(b["counts"])
    n, r = b["n_rows"], b["n_islands"]
    assert r > 0
    assert torch.equal(a["outputs"].hdr[: 3 * r], b["outputs"].hdr[: 3 * r])
    assert torch.equal(a["outputs"].pool[:n], b["outputs"].pool[:n])
    assert torch.equal(a["outputs"].pedestal, b["outputs"].pedestal) and torch.equal(a["q"], b["q"])
