"""The phased form of the default call (count and compaction in one launch, from some
2,000 tiles on, or a few hundred with wide windows): bit-exact against the two-pass
form (grid > 0 asks for it) and, where the input is small, against the oracle."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

TWO_PASS = 200  # CTAs per kernel
NOMINAL = dict(threshold=30, pre=8, post=24, decim=(32,))
WIDE = dict(threshold=25, pre=8, post=64, decim=(8, 100))
WIDER = dict(threshold=25, pre=30, post=60, decim=(32,))


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


def draw(torch, F, C, X, N, seed, rate=0.004):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    x = torch.randint(-1, 2, (F, C, X, N), generator=g, device="cuda", dtype=torch.int16)
    x += (torch.rand((F, C, 1, N), generator=g, device="cuda") < rate).to(torch.int16) * 300
    x[:, :, 1] += 111  # a pedestal
    return x


def run(env, x, lens, grid, rows, hdrs, **kw):
    torch, daq = env["torch"], env["daq"]
    F, C, X, N = x.shape
    out = daq.Outputs(torch, "cuda", F, C, X, hdrs, rows)
    out.pool.fill_(-12345)
    out.hdr.fill_(-7)
    r = daq.process_fills(x, fill_len=lens, grid=grid, outputs=out, allow=(daq.DAQ_ECAPACITY,), **kw)
    return r["status"], r["counts"], out.hdr, out.pool, out.pedestal, r["q"]


# just over the line of 14 tiles an SM (ragged last tile, ragged last chunk), then ranges of each parameter
@pytest.mark.parametrize("F,C,X,N,lens,params,rate", [
    (1, 4, 54, 239_000, None, NOMINAL, 0.004),
    (1, 5, 56, 191_112, None, dict(NOMINAL, pre=0, post=0), 0.004),
    (1, 4, 40, 252_000, None, dict(NOMINAL, pre=16, post=100), 0.002),
    (3, 4, 54, 100_008, [100_008, 0, 77], NOMINAL, 0.004),
    (3, 4, 54, 100_008, [449, 448, 100_001], NOMINAL, 0.004),
    (64, 5, 54, 3_200, list(range(3_200, 0, -50)), NOMINAL, 0.004),
    (2, 4, 54, 140_000, [0, 0], NOMINAL, 0.004),
    (2, 4, 54, 140_000, [5, 3], NOMINAL, 0.004),
    (2, 4, 54, 140_000, None, dict(NOMINAL, threshold=-30_000), 0.0),
    (2, 4, 54, 140_000, None, dict(NOMINAL, threshold=30_000), 0.0),
    (1, 4, 48, 239_000, None, dict(NOMINAL, decim=(100, 7), ped_samples=1000), 0.03),
    (1, 24, 54, 140_000, None, NOMINAL, 0.0005),
    (1, 4, 2, 239_000, None, dict(NOMINAL, threshold=100, decim=(8,)), 0.004),
    (2, 7, 4, 70_000, [70_000, 69_999], NOMINAL, 0.004),
    (1, 12, 22, 80_648, None, dict(NOMINAL, decim=(100,)), 0.004),
    (1, 4, 36, 250_000, None, WIDE, 0.001),
])
def test_matches_two_pass(env, F, C, X, N, lens, params, rate):
    torch, daq = env["torch"], env["daq"]
    x = draw(torch, F, C, X, N, seed=N + X, rate=rate)
    for flags, share in ((0, 1.0), (daq.DAQ_DEBUG_CHECKS, 1.0), (0, 0.4)):
        rows, hdrs = int(F * C * N * share) + 64, int(F * C * N * share / 2) + 64
        if share < 1:  # too few records and rows for most inputs
            rows, hdrs = rows // 8, hdrs // 64
        a = run(env, x, lens, 0, rows, hdrs, flags=flags, fill_base=3, calo_base=1, q_calos=C + 2, **params)
        b = run(env, x, lens, TWO_PASS, rows, hdrs, flags=flags, fill_base=3, calo_base=1, q_calos=C + 2, **params)
        assert a[0] == b[0] and list(a[1]) == list(b[1])
        for u, v in zip(a[2:], b[2:]):
            assert torch.equal(u, v)


@pytest.mark.parametrize("X,params", [(54, WIDE), (40, WIDE), (54, WIDER), (56, WIDER)])
@pytest.mark.parametrize("N,lens", [(35_000, None), (34_728, [34_728, 11_000]), (35_840, [35_840, 0])])
def test_wide_windows_match_oracle(env, X, params, N, lens):
    """post = 64: from 2 tiles an SM on (48 crystals; 40 stay with the two-pass form)."""
    torch, oracle, daq = env["torch"], env["oracle"], env["daq"]
    x = draw(torch, 2, 2, X, N, seed=X + N, rate=0.002)
    ref = oracle.process_fills(x.cpu().numpy(), params, fill_len=lens, n_threads=8)
    r = daq.process_fills(x, fill_len=lens, **params)
    o = r["outputs"]
    assert r["status"] == daq.DAQ_OK and r["n_islands"] == ref["n_islands"] > 20 and r["n_rows"] == ref["n_rows"]
    assert np.array_equal(o.islands_host(r["n_islands"]), ref["islands"])
    assert np.array_equal(o.pool[: r["n_rows"]].cpu().numpy(), ref["pool"])
    assert np.array_equal(o.pedestal.cpu().numpy(), ref["pedestal"])
    assert np.array_equal(r["q"].cpu().numpy(), ref["q"])


def test_captured_and_on_several_streams(env):
    """Calls on three streams at once, each with its own workspace, then one captured
    in a graph and replayed."""
    torch, daq = env["torch"], env["daq"]
    F, C, X, N = 1, 4, 54, 239_000
    xs = [draw(torch, F, C, X, N, seed=s) for s in range(3)]
    refs = [run(env, x, None, TWO_PASS, C * N, C * N, **NOMINAL) for x in xs]
    streams = [torch.cuda.Stream() for _ in xs]
    nq = refs[0][5].numel()
    outs = [daq.Outputs(torch, "cuda", F, C, X, C * N, C * N) for _ in xs]
    qs = [torch.zeros(nq, dtype=torch.int64, device="cuda") for _ in xs]
    ws = [torch.empty(daq.daq_workspace_size(C, X, N, F, daq.make_params(**NOMINAL)), dtype=torch.uint8, device="cuda")
          for _ in xs]
    torch.cuda.synchronize()
    for _ in range(5):
        for x, o, q, w, s in zip(xs, outs, qs, ws, streams):
            daq.process_fills(x, q=q, outputs=o, workspace=w, stream=s, sync=False, **NOMINAL)
    torch.cuda.synchronize()
    for o, q, ref in zip(outs, qs, refs):
        n, m = int(ref[1][0]), int(ref[1][1])
        assert o.counts.tolist() == list(ref[1])
        assert torch.equal(o.hdr[: 3 * n], ref[2][: 3 * n]) and torch.equal(o.pool[:m], ref[3][:m])
        assert torch.equal(q.view(-1), 5 * ref[5].view(-1))
    g = torch.cuda.CUDAGraph()
    qs[0].zero_()
    outs[0].pool.zero_()
    torch.cuda.synchronize()
    with torch.cuda.graph(g):
        daq.process_fills(xs[0], q=qs[0], outputs=outs[0], workspace=ws[0], stream=torch.cuda.current_stream(), sync=False,
                          **NOMINAL)
    for _ in range(2):
        g.replay()
    torch.cuda.synchronize()
    m = int(refs[0][1][1])
    assert torch.equal(outs[0].pool[:m], refs[0][3][:m]) and torch.equal(qs[0].view(-1), 2 * refs[0][5].view(-1))
