"""daq_crystal_sum of fills far shorter than their rows: exact, and no sample past a
fill's length is paid for."""
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
    import oracle
    import paper_1611_04959_gb300 as daq
    return dict(torch=torch, oracle=oracle, daq=daq)


@pytest.mark.parametrize("N", [64, 800, 801])
@pytest.mark.parametrize("lens", [[0], [1], [7, 8, 9], [0, 16, 800, 15, 3]])
def test_matches_oracle(env, N, lens):
    torch, daq, oracle = env["torch"], env["daq"], env["oracle"]
    lens = np.minimum(np.array(lens, np.int32), N)
    s = np.random.default_rng(N).integers(-3000, 4096, size=(len(lens), 2, 5, N)).astype(np.int16)
    want = oracle.crystal_sum(s, fill_len=lens, ped_samples=6)
    got = daq.crystal_sum(torch.from_numpy(s).cuda(), ped_samples=6, fill_len=lens)
    assert np.array_equal(got.cpu().numpy(), want)


def test_short_fills_cost_the_accumulators_alone(env):
    """Eight fills, each a tenth of its rows: the accumulators' 16 bytes a cell and 1.6
    of samples, against 32 for whole fills - 0.55 of the time by bytes.  Reading every
    sample would make it 0.9 or more; the line is half way."""
    torch, daq = env["torch"], env["daq"]
    F, C, X, N = 8, 24, 54, 70_000
    x = torch.randint(1700, 1900, (F, C, X, N), dtype=torch.int16, device="cuda")
    q = torch.zeros((C, X, N), dtype=torch.int64, device="cuda")
    ws = torch.empty(daq.daq_crystal_sum_workspace_size(C, X, F), dtype=torch.uint8, device="cuda")

    def ms(lens):
        ts = []
        for _ in range(9):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            daq.crystal_sum(x, q=q, fill_len=lens, workspace=ws, sync=False)
            b.record()
            torch.cuda.synchronize()
            ts.append(a.elapsed_time(b))
        return sorted(ts)[4]

    short = torch.full((F,), N // 10, dtype=torch.int32, device="cuda")
    assert ms(short) < 0.72 * ms(None)
