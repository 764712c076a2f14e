"""Rows that share no 16-byte alignment (a row pitch that is not a multiple of 8
samples, or an input that starts between 16-byte boundaries): the two-pass form
copies each tile row by row.  Bit-exact against the oracle, with the input's two
ends at every phase, windows on both count passes, uneven fills and every tile
width."""
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


NOMINAL = dict(threshold=30, pre=8, post=24, decim=(32,))
WIDE = dict(threshold=25, pre=8, post=64, decim=(8, 100))
EDGE = dict(threshold=40, pre=0, post=0, decim=(7,))


@pytest.mark.parametrize("shift", [0, 1, 2, 7])
@pytest.mark.parametrize("N", [1, 5, 448, 449, 900, 2047, 6001, 6002, 6004])
@pytest.mark.parametrize("X,params,tile", [(54, NOMINAL, 0), (54, WIDE, 0), (1, EDGE, 128), (33, NOMINAL, 224), (64, NOMINAL, 0),
                                           (63, WIDE, 384)])
def test_matches_oracle(env, N, X, params, tile, shift):
    torch, oracle, daq = env["torch"], env["oracle"], env["daq"]
    rng = np.random.default_rng(N * 64 + X + shift)
    F, C = 2, 2
    s = rng.integers(-6, 7, size=(F, C, X, N)).astype(np.int16)
    s[rng.random(s.shape) < 0.002] += 300
    s[rng.random(s.shape) < 1e-4] = rng.choice([-32768, 32767])
    lens = None if N % 2 == 0 else np.array([N, max(0, N - 9)], np.int32)
    ref = oracle.process_fills(s, params, fill_len=lens)
    # only the samples themselves are allocated past `shift` elements: a read outside them would show in a checker
    flat = torch.empty(shift + s.size, dtype=torch.int16, device="cuda")
    flat[shift:] = torch.from_numpy(s.reshape(-1))
    x = flat[shift:].view(F, C, X, N)
    for flags in (0, daq.DAQ_SPARSE):
        r = daq.process_fills(x, fill_len=lens, tile=tile, flags=flags, **params)
        o = r["outputs"]
        assert r["status"] == daq.DAQ_OK and r["n_islands"] == ref["n_islands"] and r["n_rows"] == ref["n_rows"]
        assert np.array_equal(o.islands_host(r["n_islands"]), ref["islands"])
        assert np.array_equal(o.pool[: r["n_rows"]].cpu().numpy(), ref["pool"])
        assert np.array_equal(o.pedestal.cpu().numpy(), ref["pedestal"])
        assert np.array_equal(r["q"].cpu().numpy(), ref["q"])
