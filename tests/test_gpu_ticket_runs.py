"""Runs of word tickets of the batched form.  In a batch that gives every warp 64
words or more, a warp draws eight consecutive word tickets at once (four from
32 words, two from 16) and decodes them one after the other.  A batch of 100
words a warp of 9 blocks an SM draws runs of eight whatever number of blocks
the kernel really has resident (up to 12 are possible)."""
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
    import paper_2310_10737_gb300 as sg
    yield torch, sg
    sg.sogrand_set_wait_limits(sg.DEFAULT_QUEUE_WAIT_US, sg.DEFAULT_LOCK_POLLS, 0)


def frames_for(torch, slot_n, words_per_warp=100):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    return words_per_warp * sms * 9 * 4 // slot_n


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
