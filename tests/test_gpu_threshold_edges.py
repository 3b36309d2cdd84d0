"""The threshold rule where its quick decision (the hardware exponential) is not
safe and the accurate functions have to decide."""
import numpy as np
import pytest

from test_gpu_mass_rounding import words
from workloads import ebch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2310_10737_gb300 as sg
    return torch, sg


# code, mean reliability, spread, {word: queries}
LARGE = [("ebch_32_26", 20000, 3, {7410: 222, 13622: 180}), ("ebch_64_57", 20000, 6, {18549: 300}),
         ("ebch_64_57", 30000, 3, {16809: 295}), ("ebch_32_26", 30000, 3, {7410: 222, 13622: 180})]


@pytest.mark.parametrize("name,mean,spread,queries", LARGE)
def test_large_masses(env, name, mean, spread, queries):
    """Log masses of tens of thousands: the accurate rule's sum moves by an ulp
    of them a list word, more than 1e-3, and its decision stands (these words
    went on past the quick decision; the query counts are the accurate rule's)."""
    torch, sg = env
    lc = ebch(name)
    x = words(lc.n, 20000, mean, spread)[list(queries)]
    c = sg.Code.from_linear_code(lc)
    out = sg.sogrand_decode(c, torch.from_numpy(x).cuda(), L=16, query_cap=300, thr=1e-3)
    torch.cuda.synchronize()
    c.close()
    assert out["queries"].tolist() == list(queries.values())
