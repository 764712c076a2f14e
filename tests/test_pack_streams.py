"""pack_pool and unpack_pool on a stream of the caller's: sizes and error words are read
once that stream has written them, whatever the current stream is doing."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


class Handle:  # all that the calls ask of a stream
    def __init__(self, stream):
        self.cuda_stream = stream.cuda_stream


@pytest.mark.parametrize("wrap", [lambda s: s, Handle], ids=["torch", "handle"])
def test_results_of_a_busy_stream(wrap):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import oracle
    import paper_1611_04959_gb300 as daq
    rng = np.random.default_rng(1)
    pool = (1800 + rng.integers(-9, 10, size=(5000, 54))).astype(np.int16)
    want = oracle.pack(pool)
    dev, packed = torch.from_numpy(pool).cuda(), torch.from_numpy(want).cuda()
    bad = packed.clone()
    bad[0] ^= 1
    daq.pack_pool(dev), daq.unpack_pool(packed, 5000, 54)       # kernels loaded
    torch.cuda.synchronize()
    side = torch.cuda.Stream()

    def busy():
        with torch.cuda.stream(side):
            torch.cuda._sleep(100_000_000)                      # some 50 ms

    for _ in range(3):
        busy()
        got, n = daq.pack_pool(dev, stream=wrap(side))
        assert n == want.size and np.array_equal(got.cpu().numpy(), want)
        busy()
        back = daq.unpack_pool(packed, 5000, 54, stream=wrap(side))
        assert np.array_equal(back.cpu().numpy(), pool)
        busy()
        with pytest.raises(daq.DaqError):
            daq.unpack_pool(bad, 5000, 54, stream=wrap(side))
    out = torch.zeros(daq.daq_pack_bound(5000, 54), dtype=torch.uint8, device="cuda")
    ws = torch.zeros(daq.daq_pack_workspace_size(5000, 54), dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    busy()
    got, n = daq.pack_pool(dev, stream=wrap(side), out=out, workspace=ws)
    assert n == want.size and got.data_ptr() == out.data_ptr() and np.array_equal(got.cpu().numpy(), want)
