"""Which form a default call takes (daq_call_form): the phased form on both sides of every
line of its rule, and that the kernel so named is what ran."""
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
    return dict(torch=torch, daq=daq, sms=torch.cuda.get_device_properties(0).multi_processor_count)


def form(env, C, X, N, F=1, at=0, **kw):
    return env["daq"].daq_call_form(1 << 20 | at, C, X, N, F, env["daq"].make_params(**kw))


def test_the_rule(env):
    daq, sms = env["daq"], env["sms"]
    many = 448 * 14 * sms                    # samples of one calorimeter: exactly 14 tiles an SM
    P, T = daq.DAQ_FORM_PHASED, daq.DAQ_FORM_TWO_PASS
    assert form(env, 1, 54, many) == P and form(env, 1, 54, many - 448) == T
    assert [form(env, 1, X, many) for X in (2, 36, 56, 58, 64, 1, 53, 55)] == [P, P, P, T, T, T, T, T]
    assert form(env, 1, 54, many + 8) == P and form(env, 1, 54, many + 4) == T          # rows of 16 bytes
    assert form(env, 1, 54, many, at=8) == T
    assert form(env, 1, 54, many // 64 // 8 * 8 + 448, F=64) == P and form(env, 1, 54, many // 64 // 8 * 8 + 448, F=65) == T
    assert form(env, 1, 54, many, flags=daq.DAQ_SPARSE) == T and form(env, 1, 54, many, flags=daq.DAQ_SKIP_ISLANDS) == T
    assert form(env, 1, 54, many, flags=daq.DAQ_SKIP_Q | daq.DAQ_DEBUG_CHECKS | daq.DAQ_SYNC) == P
    assert form(env, 1, 54, many, wait_limit_ns=10 ** 9) == P and form(env, 1, 54, many, wait_limit_ns=10 ** 9 - 1) == T
    assert form(env, 1, 54, many, tile=448) == P and form(env, 1, 54, many, tile=384) == T
    assert form(env, 1, 54, many, pre=30, post=60) == P and form(env, 1, 54, many, pre=16, post=100) == T
    few = 448 * 2 * sms                      # wide windows: two tiles an SM, from 48 crystals on
    assert form(env, 1, 54, few, post=64) == P and form(env, 1, 54, few - 448, post=64) == T
    assert form(env, 1, 48, few, post=64) in (P, T) and form(env, 1, 40, few, post=64) == T
    assert [form(env, 1, 54, many, grid=g) for g in (200, -1, -2, -3, -4, -5, -6)] == \
        [T, daq.DAQ_FORM_PLAIN, daq.DAQ_FORM_PLAIN, daq.DAQ_FORM_PIPELINED, daq.DAQ_FORM_SINGLE_LAUNCH, daq.DAQ_FORM_STREAM,
         daq.DAQ_FORM_SINGLE_READ]
    assert form(env, 1, 54, many + 4, grid=-5) == T and form(env, 1, 53, many, grid=-6) == T
    assert form(env, 1, 54, many, grid=-7) == daq.DAQ_EINVAL and form(env, 1, 65, many) == daq.DAQ_EUNSUPPORTED


# the shapes of test_phased.py that are meant to be phased, and the two that are not
@pytest.mark.parametrize("F,C,X,N,kw,phased", [
    (1, 4, 54, 239_000, {}, True), (1, 5, 56, 191_112, dict(pre=0, post=0), True),
    (1, 4, 40, 252_000, dict(pre=16, post=100), False), (3, 4, 54, 100_008, {}, True), (64, 5, 54, 3_200, {}, True),
    (2, 4, 54, 140_000, {}, True), (1, 4, 48, 239_000, dict(decim=(100, 7), ped_samples=1000), True),
    (1, 24, 54, 140_000, {}, True), (1, 4, 2, 239_000, dict(decim=(8,)), True), (2, 7, 4, 70_000, {}, True),
    (1, 12, 22, 80_648, dict(decim=(100,)), True), (1, 4, 36, 250_000, dict(post=64, decim=(8, 100)), True),
    (2, 2, 54, 35_000, dict(post=64, decim=(8, 100)), True), (2, 2, 40, 35_000, dict(post=64, decim=(8, 100)), False),
    (2, 2, 54, 35_000, dict(pre=30, post=60), True), (2, 2, 56, 34_728, dict(pre=30, post=60), True)])
def test_shapes_meant_to_be_phased_are(env, F, C, X, N, kw, phased):
    if env["sms"] != 152:
        pytest.skip("the shapes are chosen for 152 SMs")
    daq = env["daq"]
    assert form(env, C, X, N, F, **kw) == (daq.DAQ_FORM_PHASED if phased else daq.DAQ_FORM_TWO_PASS)


@pytest.mark.parametrize("grid,phased", [(0, True), (200, False)])
def test_what_ran(env, grid, phased):
    """The phased kernel publishes a word for each tile in a part of the workspace that the
    two-pass form does not touch."""
    torch, daq = env["torch"], env["daq"]
    C, X, N = 4, 54, 448 * 14 * env["sms"] // 4 // 8 * 8 + 448
    x = torch.randint(1790, 1811, (1, C, X, N), device="cuda", dtype=torch.int16)
    ws = torch.zeros(daq.daq_workspace_size(C, X, N, 1, daq.make_params()), dtype=torch.uint8, device="cuda")
    assert daq.daq_call_form(x.data_ptr(), C, X, N, 1, daq.make_params(grid=grid)) == \
        (daq.DAQ_FORM_PHASED if phased else daq.DAQ_FORM_TWO_PASS)
    daq.process_fills(x, workspace=ws, grid=grid)

    def up(v):
        return -(-v // 256) * 256

    words = up(up(up(512 + 8 * 2) + 4) + 4 * C)
    there = ws[words: words + 4 * C * -(-N // 448)].view(torch.int32)
    assert bool((there < 0).all()) if phased else bool((there == 0).all())   # bit 31: published
