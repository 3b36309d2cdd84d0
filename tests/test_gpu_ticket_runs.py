"""Runs of word tickets of the batched form.  In a batch that gives every warp 64
words or more, a warp draws eight consecutive word tickets at once (four from
32 words, two from 16) and decodes them one after the other.  A batch of 100
words a warp of 9 blocks an SM draws runs of eight whatever number of blocks
the kernel really has resident (up to 12 are possible)."""
import numpy as np
import pytest

from workloads import awgn_frames, ebch, shorten

pytestmark = pytest.mark.gpu
OUT = ("bits", "half_iters", "status", "queries", "par_queries", "weight_sum")


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2310_10737_gb300 as sg
    yield torch, sg
    sg.sogrand_set_wait_limits(sg.DEFAULT_QUEUE_WAIT_US, sg.DEFAULT_LOCK_POLLS, 0)


def frames_for(torch, slot_n, words_per_warp=100):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    return words_per_warp * sms * 9 * 4 // slot_n


def zero_frames(torch, F, nc, nr, rate, ebn0, seed):
    """Channel LLRs of F all-zero codewords (the decoder is the same for all of a linear code's)."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    s2 = 1.0 / (2.0 * rate * 10.0 ** (ebn0 / 10.0))
    return (2.0 / s2) * (1.0 + s2 ** 0.5 * torch.randn((F, nc, nr), generator=g, device="cuda"))


def test_wait_limit_covers_a_run(env):
    """A wait limit that is enough for one word at a time is enough for warps
    that hold eight: equal searches to the cap (lists that never fill), whose
    last runs the other warps wait for."""
    torch, sg = env
    n, m, cap = 64, 32, 65536
    H = np.concatenate([np.random.default_rng(1).integers(0, 2, (m, n - m), dtype=np.uint8), np.eye(m, dtype=np.uint8)], 1)
    H[-1] = 1
    c = sg.Code(H)
    c.reserve(cap)
    F = frames_for(torch, n, 85)
    d = torch.randn((F, n, n), generator=torch.Generator(device="cuda").manual_seed(5), device="cuda")
    sg.sogrand_set_wait_limits(1500, -1, -1)
    try:
        o = sg.product_decode(c, d, L=4, query_cap=cap, max_iter=1, persistent=True)
    finally:
        sg.sogrand_set_wait_limits(sg.DEFAULT_QUEUE_WAIT_US, -1, -1)
        c.close()
    assert (o["queries"] == 2 * n * cap).all()


@pytest.mark.parametrize("row,col,thr", [("ebch_64_57", "ebch_64_57", 1e-4), ("ebch_64_57", "ebch_64_51", 1e-5),
                                         ("ebch_32_26", "ebch_16_11", 0.0), ("ebch_16_11", "ebch_32_26", 1e-4)])
def test_runs_of_eight_equal_plain_form(env, row, col, thr):
    """Threshold rule, two codes, and codes of different lengths (a half of the
    shorter kind leaves half of its tickets unused)."""
    torch, sg = env
    r, c = ebch(row), ebch(col)
    F = frames_for(torch, max(r.n, c.n))
    d = zero_frames(torch, F, c.n, r.n, r.k * c.k / (r.n * c.n), 2.75, 11)
    kr = sg.Code.from_linear_code(r)
    kc = kr if row == col else sg.Code.from_linear_code(c)
    a = sg.product_decode(kr, d, query_cap=3000, thr=thr, max_iter=6, col_code=kc)
    b = sg.product_decode(kr, d, query_cap=3000, thr=thr, max_iter=6, col_code=kc, persistent=True)
    torch.cuda.synchronize()
    assert (a["half_iters"] > 2).any()
    for key in OUT:
        assert torch.equal(a[key], b[key]), key


def test_runs_of_eight_wrapped_diagonals(env):
    """A QC-GLDPC batch in one call against the same frames in eight calls of small batches (single tickets)."""
    torch, sg = env
    lc = ebch("ebch_32_26")
    c = sg.Code.from_linear_code(lc)
    F = frames_for(torch, lc.n)
    d = zero_frames(torch, F, lc.n, lc.n, 2 * lc.k / lc.n - 1, 2.5, 12)
    p = dict(query_cap=3000, thr=1e-5, max_iter=6)
    big = sg.gldpc_decode(c, d, **p)
    small = [sg.gldpc_decode(c, x, **p) for x in d.chunk(8)]
    torch.cuda.synchronize()
    for key in OUT[:5]:
        assert torch.equal(big[key], torch.cat([s[key] for s in small])), key
    c.close()


def test_runs_of_eight_through_the_server(env):
    """One request large enough for runs, parked and resumed every two halves, against the plain form."""
    torch, sg = env
    lc = ebch("ebch_32_26")
    c = sg.Code.from_linear_code(lc)
    F = frames_for(torch, lc.n)
    d = zero_frames(torch, F, lc.n, lc.n, (lc.k / lc.n) ** 2, 2.5, 13)
    p = dict(L=4, query_cap=3000, thr=1e-4, alpha=0.5, max_iter=6)
    ref = sg.product_decode(c, d, **p)
    assert (ref["half_iters"] > 4).any()  # more than two epochs
    s = sg.Server([c], [F], epoch_halves=2, **p)
    ticket, out = s.submit(0, d.cpu().pin_memory())
    assert s.wait(ticket)[0]
    s.close()
    for key in OUT[:4]:
        np.testing.assert_array_equal(np.asarray(out[key]).ravel(), ref[key].cpu().numpy().ravel(), err_msg=key)
    c.close()


@pytest.mark.parametrize("srow,scol", [(3, 3), (3, 5), (5, 0)])
def test_bits_of_ragged_widths(env, srow, scol):
    """Rows that do not start on byte boundaries, after row and after column
    halves: the decoded frames are the ones sent, bit by bit."""
    torch, sg = env
    base = ebch("ebch_32_26")
    r, c = shorten(base, srow), shorten(base, scol)
    _, X, llr = awgn_frames(r, 300, 3.25, seed=14, col_code=c)
    kr, kc = sg.Code.from_linear_code(r), sg.Code.from_linear_code(c)
    for persistent in (False, True):
        o = sg.product_decode(kr, torch.from_numpy(llr).cuda(), max_iter=10, col_code=kc, persistent=persistent)
        torch.cuda.synchronize()
        got = sg.unpack_bits(o["bits"], c.n, r.n)
        hit = (got == X).reshape(300, -1).all(1)
        half, ok = o["half_iters"].cpu().numpy(), o["status"].cpu().numpy() == 0
        for parity in (0, 1):
            sel = ok & (half % 2 == parity)
            assert sel.sum() >= 20 and hit[sel].mean() >= 0.95
