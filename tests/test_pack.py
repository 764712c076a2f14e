"""GPU lossless packing of pool rows (daq_pack_pool / daq_unpack_pool) against
the oracle's encoder and decoder: the streams must be byte-identical, and
decoding must give the pool back exactly, for ragged sizes (partial last
block, block counts on and around the scan's chunk boundary), every crystal
count up to 64, extreme sample values, the benchmark fill's own pool, short
output capacity and damaged streams."""
import numpy as np
import pytest


@pytest.fixture(scope="module")
def daq():
    from paper_1611_04959_gb300 import build
    build.build()
    import paper_1611_04959_gb300 as d
    return d


def test_bounds_and_argument_checks(daq):
    assert daq.daq_pack_bound(0, 54) == 24
    assert daq.daq_pack_bound(33, 2) == 16 + 8 * 3 + 2 * 2 * 4 * 18
    assert daq.daq_pack_bound(10, 65) == -1 and daq.daq_pack_bound(-1, 5) == -1
    assert daq.daq_pack_workspace_size(1000, 54) > 0
    assert daq.daq_pack_pool(0, 0, 65, 0, 0, 8, 0, 0, None) == daq.DAQ_EUNSUPPORTED     # n_xtal > 64
    assert daq.daq_pack_pool(0, 10, 4, 0, 0, None, 0, 0, None) == daq.DAQ_EINVAL      # no out_bytes
    assert daq.daq_pack_pool(2, 10, 4, 16, 1000, 8, 16, 4096, None) == daq.DAQ_EINVAL  # pool not 16-byte aligned
    assert daq.daq_unpack_pool(None, 100, 10, 4, 0, 0, None) == daq.DAQ_EINVAL


@pytest.fixture(scope="module")
def env(daq):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import oracle
    return dict(torch=torch, oracle=oracle, daq=daq)


CASES = [(0, 3), (1, 1), (31, 2), (32, 54), (33, 54), (1000, 5), (4097, 3), (32 * 1024, 2), (32 * 1024 + 5, 7),
         (32 * 2048, 1), (777, 64), (500, 63)]


@pytest.mark.gpu
@pytest.mark.parametrize("rows,X", CASES)
def test_stream_matches_oracle_and_round_trips(env, rows, X):
    torch, daq, oracle = env["torch"], env["daq"], env["oracle"]
    rng = np.random.default_rng(rows * 131 + X)
    if rows % 3 == 0:
        pool = rng.integers(-32768, 32768, size=(rows, X))
    else:
        pool = 1800 + np.cumsum(rng.integers(-6, 7, size=(rows, X)), axis=0)
    pool = np.asarray(pool).astype(np.int16)
    want = oracle.pack(pool)
    dev = torch.from_numpy(pool).cuda() if rows else torch.zeros((1, X), dtype=torch.int16, device="cuda")
    got, n = daq.pack_pool(dev, rows)
    assert n == want.size
    assert np.array_equal(got.cpu().numpy(), want)
    back = daq.unpack_pool(got, rows, X)
    assert np.array_equal(back.cpu().numpy(), pool)
    back2 = daq.unpack_pool(torch.from_numpy(want).cuda(), rows, X)       # the oracle's stream decodes too
    assert np.array_equal(back2.cpu().numpy(), pool)


@pytest.mark.gpu
def test_crystal_counts_in_any_order(env):
    """The packing kernels size their shared memory by the crystal count: calls
    with a large, a small and again the large count, in one process, all run
    and match the oracle (a smaller call must not lower the kernels' limit)."""
    torch, daq, oracle = env["torch"], env["daq"], env["oracle"]
    for k, (rows, X) in enumerate([(4000, 64), (300, 1), (70, 2), (4000, 64), (1000, 54), (33, 3), (1000, 54)]):
        rng = np.random.default_rng(900 + k)
        pool = (1800 + np.cumsum(rng.integers(-9, 10, size=(rows, X)), axis=0)).astype(np.int16)
        got, n = daq.pack_pool(torch.from_numpy(pool).cuda(), rows)
        assert np.array_equal(got.cpu().numpy(), oracle.pack(pool)), (rows, X)


@pytest.mark.gpu
@pytest.mark.parametrize("rows,X", [(777, 54), (4096 + 13, 7), (2000, 64), (1500, 9)])
def test_every_width_class_and_mix(env, rows, X):
    """Columns whose row-to-row steps span every width class: <= 7 bits (four
    columns per transpose), 8-15 (pairs), 16-17 (alone), in every mix along a
    row, so each group size meets each fallback."""
    torch, daq, oracle = env["torch"], env["daq"], env["oracle"]
    rng = np.random.default_rng(rows * 7 + X)
    scale = 2 ** (np.arange(X) * 5 % 17)                     # step sizes 1 .. 65536 across the columns
    steps = rng.integers(-1, 2, size=(rows, X)) * rng.integers(0, scale + 1, size=(rows, X))
    pool = (np.cumsum(steps, axis=0) % 65536 - 32768).astype(np.int16)
    want = oracle.pack(pool)
    got, n = daq.pack_pool(torch.from_numpy(pool).cuda(), rows)
    assert n == want.size and np.array_equal(got.cpu().numpy(), want)
    assert np.array_equal(daq.unpack_pool(got, rows, X).cpu().numpy(), pool)
    assert np.array_equal(daq.unpack_pool(torch.from_numpy(want).cuda(), rows, X).cpu().numpy(), pool)


@pytest.mark.gpu
def test_full_fill_pool(env):
    torch, daq, oracle = env["torch"], env["daq"], env["oracle"]
    import synth
    from synth import workloads as W
    w = W.PLAIN_FULL_FILL
    s = synth.generate(w.config())
    res = daq.process_fills(torch.from_numpy(s).cuda(), **w.params())
    rows = res["n_rows"]
    pool = res["outputs"].pool[:rows]
    got, n = daq.pack_pool(pool, rows)
    host_pool = pool.cpu().numpy()
    want = oracle.pack(host_pool)
    assert n == want.size and np.array_equal(got.cpu().numpy(), want)
    assert np.array_equal(daq.unpack_pool(got, rows, 54).cpu().numpy(), host_pool)
    assert host_pool.nbytes / n > 2.0          # noise-dominated rows: a few bits per sample


@pytest.mark.gpu
def test_short_capacity_and_damaged_streams(env):
    torch, daq, oracle = env["torch"], env["daq"], env["oracle"]
    rng = np.random.default_rng(4)
    pool = (1800 + np.cumsum(rng.integers(-4, 5, size=(300, 6)), axis=0)).astype(np.int16)
    want = oracle.pack(pool)
    dev = torch.from_numpy(pool).cuda()
    cap = want.size // 2
    out = torch.full((want.size + 64,), 0xAB, dtype=torch.uint8, device="cuda")
    ws = torch.empty(daq.daq_pack_workspace_size(300, 6), dtype=torch.uint8, device="cuda")
    nbytes = torch.zeros(1, dtype=torch.int64, device="cuda")
    rc = daq.daq_pack_pool(dev.data_ptr(), 300, 6, out.data_ptr(), cap, nbytes.data_ptr(), ws.data_ptr(), ws.numel(),
                           None)
    assert rc == daq.DAQ_OK
    torch.cuda.synchronize()
    assert int(nbytes.item()) == want.size                   # the size needed
    o = out.cpu().numpy()
    assert np.array_equal(o[:cap], want[:cap]) and (o[cap:] == 0xAB).all()
    with pytest.raises(daq.DaqError):                         # cut short
        daq.unpack_pool(torch.from_numpy(want[: want.size - 8]).cuda(), 300, 6)
    with pytest.raises(daq.DaqError):                         # header does not match
        daq.unpack_pool(torch.from_numpy(want).cuda(), 299, 6)


def _relocated(stream, rows, X, kind, rng):
    """A stream that decodes to the same rows with its blocks' payloads in
    another place: in reverse order, with gaps between them, or with every
    offset but a block's own made useless as the end of the block before it."""
    nb = -(-rows // 32)
    head = 16 + 8 * (nb + 1)
    offs = stream[16:head].view("<u8").astype(np.int64)
    blocks = [stream[head + offs[b]: head + offs[b + 1]] for b in range(nb)]
    out, at = [], np.zeros(nb + 1, np.int64)
    order = range(nb - 1, -1, -1) if kind == "reversed" else range(nb)
    pos = 0
    for b in order:
        if kind == "gaps":
            out.append(rng.integers(0, 256, 4 * int(rng.integers(0, 40)), dtype=np.uint8))
            pos += out[-1].size
        at[b] = pos
        out.append(blocks[b])
        pos += blocks[b].size
    at[nb] = pos
    if kind == "shared":              # two equal blocks kept once: the next offset lies before the block's end
        for b in range(1, nb):
            if np.array_equal(blocks[b], blocks[b - 1]):
                at[b] = at[b - 1]
    payload = np.concatenate(out)
    return np.concatenate([stream[:16], at.astype("<u8").view(np.uint8), payload])


@pytest.mark.gpu
@pytest.mark.parametrize("X", [1, 9, 16, 20, 31, 33, 54, 64])
@pytest.mark.parametrize("kind", ["plain", "reversed", "gaps", "shared"])
def test_decoder_follows_any_valid_offsets(env, X, kind):
    """Crystal counts that put several blocks side by side in a warp, ragged
    last blocks, narrow and wide columns in one block, and offset tables that a
    decoder must follow although the blocks do not lie back to back."""
    torch, daq, oracle = env["torch"], env["daq"], env["oracle"]
    rng = np.random.default_rng(31 * X + len(kind))
    rows = 32 * 41 + 13
    pool = 1800 + np.cumsum(rng.integers(-5, 6, size=(rows, X)), axis=0)
    wide = rng.integers(0, rows, 40)
    pool[wide, rng.integers(0, X, 40)] += rng.integers(-30000, 30000, 40)
    if kind == "shared":
        pool[64:96] = pool[32:64]
        pool[96:128] = pool[32:64]
    pool = pool.astype(np.int16)
    stream = oracle.pack(pool)
    if kind != "plain":
        stream = _relocated(stream, rows, X, kind, rng)
    assert np.array_equal(oracle.unpack(stream, rows, X), pool)
    got = daq.unpack_pool(torch.from_numpy(stream).cuda(), rows, X)
    assert np.array_equal(got.cpu().numpy(), pool)
    bad = stream.copy()               # a width no encoder writes, in the last block
    nb = -(-rows // 32)
    off = int(bad[16 + 8 * (nb - 1): 24 + 8 * (nb - 1)].view("<u8")[0])
    bad[16 + 8 * (nb + 1) + off + 2] = 18
    with pytest.raises(daq.DaqError):
        daq.unpack_pool(torch.from_numpy(bad).cuda(), rows, X)


@pytest.mark.gpu
def test_many_chunks_of_every_kind(env):
    """Enough blocks that every CTA of the encoder takes many turns, with
    stretches of noise, of steps past a byte, and of full-range samples whose
    words fit no stage and are encoded again into place."""
    torch, daq, oracle = env["torch"], env["daq"], env["oracle"]
    rng = np.random.default_rng(77)
    rows, X = 900_007, 33
    pool = 1800 + rng.integers(-9, 10, size=(rows, X))
    for k in range(0, rows, 40_000):
        n = int(rng.integers(1, 6_000))
        pool[k: k + n] += rng.integers(-600, 600, size=pool[k: k + n].shape) * (rng.random(pool[k: k + n].shape) < 0.05)
        pool[k + 10_000: k + 10_000 + n] = rng.integers(-32768, 32768, size=pool[k + 10_000: k + 10_000 + n].shape)
    pool = pool.astype(np.int16)
    want = oracle.pack(pool)
    dev = torch.from_numpy(pool).cuda()
    for _ in range(2):
        got, n = daq.pack_pool(dev)
        assert n == want.size and np.array_equal(got.cpu().numpy(), want)
    assert np.array_equal(daq.unpack_pool(got, rows, X).cpu().numpy(), pool)
