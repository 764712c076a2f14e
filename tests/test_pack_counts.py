"""daq_pack_pool and daq_unpack_pool at every crystal count that they take, in rising
and in falling order in one process: the kernels' shared-memory limit is set once and
has to hold for whichever count asks for most."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("counts", [range(1, 65), range(64, 0, -1)], ids=["rising", "falling"])
def test_every_crystal_count(counts):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import oracle
    import paper_1611_04959_gb300 as daq
    for X in counts:
        rng = np.random.default_rng(X)
        rows = 32 * 150 + 7                      # two chunks at X = 4 (128 blocks each), more above
        pool = 1800 + rng.integers(-9, 10, size=(rows, X))
        pool[rng.integers(0, rows, 40), rng.integers(0, X, 40)] += 900
        pool = pool.astype(np.int16)
        want = oracle.pack(pool)
        got, n = daq.pack_pool(torch.from_numpy(pool).cuda())
        assert n == want.size and np.array_equal(got.cpu().numpy(), want), X
        assert np.array_equal(daq.unpack_pool(got, rows, X).cpu().numpy(), pool), X
