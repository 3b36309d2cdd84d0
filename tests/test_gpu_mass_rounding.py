"""Remaining mass summed directly (the cost DP): the same word gives the same
bits in every kernel that the sum is compiled into, with and without the
threshold rule.  Its products with the cost scale are rounded by themselves and
log2(sum) - gamma C* once; where the compiler was free to choose, p_miss moved
by up to 5e-6 relative at ordinary reliabilities (an ulp of the log mass) and by
2e-3 at log masses of 20,000.  Inputs are multiples of 1/256, so that they
are the same everywhere; the golden bits are p_miss's."""
import os

import numpy as np
import pytest

from workloads import ebch

pytestmark = pytest.mark.gpu

GOLDEN = os.path.join(os.path.dirname(__file__), "golden", "remaining_mass_bits.txt")
# code, words, query cap, list size, threshold, mean reliability, spread
CASES = [("ebch_64_57", 2000, 200, 4, 0.0, 20, 6), ("ebch_64_51", 2000, 200, 4, 0.0, 20, 6),
         ("ebch_32_26", 2000, 31, 16, 0.0, 50, 3), ("ebch_128_120", 2000, 200, 4, 0.0, 20, 6),
         ("ebch_32_26", 20000, 300, 16, 1e-3, 20000, 3), ("ebch_64_57", 20000, 300, 16, 1e-3, 30000, 3)]


def words(n, count, mean, spread):
    """|lambda| = mean + k / 256, k the sum of three uniform integers, about two signs flipped."""
    r = np.random.default_rng(7)
    k = r.integers(-256 * spread, 256 * spread + 1, (3, count, n)).sum(0)
    s = 1 - 2 * (r.integers(0, n, (count, n)) < 2)
    return ((mean + k / 256.0) * s).astype(np.float32)


@pytest.mark.parametrize("case", range(len(CASES)))
def test_p_miss_bits(case):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2310_10737_gb300 as sg
    name, count, cap, L, thr, mean, spread = CASES[case]
    rows = [ln.split() for ln in open(GOLDEN) if not ln.startswith("#")]
    rows = [(int(w), int(b, 16), int(q)) for c, w, b, q in rows if int(c) == case]
    assert len(rows) >= 12
    lc = ebch(name)
    x = words(lc.n, count, mean, spread)[[w for w, _, _ in rows]]
    c = sg.Code.from_linear_code(lc)
    out = sg.sogrand_decode(c, torch.from_numpy(x).cuda(), L=L, query_cap=cap, thr=thr)
    torch.cuda.synchronize()
    c.close()
    np.testing.assert_array_equal(out["queries"].cpu().numpy(), [q for _, _, q in rows])
    np.testing.assert_array_equal(out["p_miss"].cpu().numpy().view(np.uint32), np.array([b for _, b, _ in rows], np.uint32))
