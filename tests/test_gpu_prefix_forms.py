"""The query loop's compact forms (prefix records with two or three trailing
ranks, then the 16-byte entries) against the oracle where they can go wrong:
query caps at chunk edges, around the ends of the two-rank (about 1000
queries) and three-rank forms (about 9000, at most 16384), orders that end
with their parity class, codes that are not even, 64-bit syndromes, and the
threshold rule, which stops a search at any listed word.  The bar is the
SISO's: queries and lists bit-exact, soft outputs within 1e-3 + 1e-4 |L|."""
import numpy as np
import pytest

from gpu_common import compare_siso
from workloads import ebch
from workloads.codes import LinearCode

pytestmark = pytest.mark.gpu


def _code(name):
    if name != "wide_syndrome":
        return ebch(name)
    rng = np.random.default_rng(3)  # n - k = 36 checks: systematic, the last one the overall parity
    n, m = 40, 36
    P = rng.integers(0, 2, (m, n - m), dtype=np.uint8)
    P[-1] = 1 ^ (P[:-1].sum(0) & 1)
    H = np.concatenate([P, np.eye(m, dtype=np.uint8)], axis=1)
    H[-1] = 1  # the sum of all rows
    G = np.concatenate([np.eye(n - m, dtype=np.uint8), P.T], axis=1)
    G[:, -1] = G[:, :-1].sum(1) & 1
    return LinearCode("wide_syndrome", n, n - m, G, H)


@pytest.mark.parametrize("name,cap,L,thr,even", [
    ("ebch_64_51", 1, 4, 0.0, True), ("ebch_64_51", 31, 4, 0.0, True), ("ebch_64_51", 32, 4, 0.0, True),
    ("ebch_64_51", 33, 4, 0.0, True), ("ebch_64_51", 863, 4, 0.0, True), ("ebch_64_51", 1025, 16, 0.0, True),
    ("ebch_64_51", 3000, 16, 0.0, True), ("ebch_64_51", 9250, 16, 0.0, True), ("ebch_64_51", 10000, 16, 1e-5, True),
    ("ebch_64_51", 17000, 16, 0.0, True), ("ebch_128_120", 10000, 16, 0.0, True),
    ("ebch_128_120", 2000, 16, 1e-4, True), ("ebch_32_26", 10000, 16, 0.0, True), ("ebch_16_7", 10000, 16, 0.0, True),
    ("ebch_8_4", 10000, 8, 0.0, True), ("ebch_8_4", 10000, 4, 1e-3, True), ("ebch_32_26", 5000, 8, 0.0, False),
    ("ebch_64_51", 2500, 3, 1e-4, False), ("wide_syndrome", 2000, 2, 0.0, True)])
def test_forms_match_oracle(oracle_lib, name, cap, L, thr, even):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2310_10737_gb300 as sg
    lc = _code(name)
    lc = LinearCode(lc.name, lc.n, lc.k, lc.G, lc.H, even=even)
    rng = np.random.default_rng(cap + L)
    # noise alone at several reliabilities (deep searches, c from 0 up), both parities
    scale = rng.choice([0.5, 2.0, 6.0], (60, 1))
    lch = (rng.standard_normal((60, lc.n)) * scale + rng.choice([-3.0, 0.0, 3.0], (60, 1))).astype(np.float32)
    c = sg.Code.from_linear_code(lc)
    out = sg.sogrand_decode(c, torch.from_numpy(lch).cuda(), L=L, query_cap=cap, thr=thr)
    torch.cuda.synchronize()
    c.close()
    ref = oracle_lib.siso_batch(oracle_lib.OracleCode(lc), lch, L=L, cap=cap, thr=thr)
    compare_siso(lc, out, ref, f"{name} cap={cap} L={L} thr={thr}")


@pytest.mark.parametrize("name", ["ebch_16_11", "ebch_32_26", "ebch_64_57", "ebch_128_120"])
def test_order_of_nearly_equal_reliabilities(oracle_lib, name):
    """The reliability sort drops the lowest bits of |lambda| from its keys and
    restores the exact order afterwards: values a few units in the last place
    apart (and equal ones, which fall to the lower index), whole words of them
    and a few among ordinary ones, must give the oracle's queries and lists."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2310_10737_gb300 as sg
    lc = ebch(name)
    rng = np.random.default_rng(12)
    W = 200
    near = np.float32(2.0) + rng.integers(0, 40, (W, lc.n)).astype(np.float32) * np.float32(2.0 ** -22)
    lch = near * rng.choice(np.array([-1.0, 1.0], np.float32), (W, lc.n))
    some = rng.random((W, lc.n)) < 0.8  # from word 100 on, most values are ordinary
    some[:100] = False
    lch = np.where(some, rng.standard_normal((W, lc.n)) * 4.0, lch).astype(np.float32)
    c = sg.Code.from_linear_code(lc)
    out = sg.sogrand_decode(c, torch.from_numpy(lch).cuda(), L=4, query_cap=3000)
    torch.cuda.synchronize()
    c.close()
    ref = oracle_lib.siso_batch(oracle_lib.OracleCode(lc), lch, L=4, cap=3000)
    compare_siso(lc, out, ref, f"{name} near ties")


@pytest.mark.parametrize("row,col,frames", [("ebch_16_11", "ebch_32_26", 1), ("ebch_16_11", "ebch_32_26", 3500),
                                            ("ebch_32_26", "ebch_16_11", 6001), ("ebch_32_26", "ebch_32_26", 12003),
                                            ("ebch_16_11", "ebch_16_11", 12001)])
def test_ticket_runs_equal_plain_form(row, col, frames):
    """Batches small and large enough that warps draw one, two, four or eight
    word tickets at once (5,472 warps: 8, 16, 32 and 64 words each), with halves
    that leave tickets unused: every output as the plain form gives it."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2310_10737_gb300 as sg
    from workloads import awgn_frames
    r, c = ebch(row), ebch(col)
    _, _, llr = awgn_frames(r, min(frames, 1500), 2.5, seed=5, col_code=c, threads=8)
    llr = np.tile(llr, (-(-frames // len(llr)), 1, 1))[:frames]
    d = torch.from_numpy(np.ascontiguousarray(llr)).cuda()
    kr, kc = sg.Code.from_linear_code(r), sg.Code.from_linear_code(c)
    kc = kr if row == col else kc
    a = sg.product_decode(kr, d, max_iter=6, col_code=kc)
    b = sg.product_decode(kr, d, max_iter=6, col_code=kc, persistent=True)
    torch.cuda.synchronize()
    for key in ("bits", "half_iters", "status", "queries", "par_queries", "weight_sum"):
        assert torch.equal(a[key], b[key]), key
