"""The threshold rule where its quick decision (the hardware exponential) is not
safe and the accurate functions have to decide."""
import numpy as np
import pytest

from gpu_common import compare_siso
from test_gpu_mass_rounding import words
from workloads import ebch
from workloads.codes import LinearCode

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


@pytest.mark.parametrize("name", ["ebch_32_26", "ebch_64_57", "ebch_128_120"])
@pytest.mark.parametrize("thr", [1e-37, 1e-40, 1e-42])
def test_denormal_thresholds(env, oracle_lib, name, thr):
    """Clean words whose miss probability is near 1e-39: a threshold of 1e-37
    stops them at the first list word, a denormal one does not (the quick sum
    overflows there)."""
    torch, sg = env
    lc = ebch(name)
    x = (45 + np.random.default_rng(3).integers(0, 1280, (40, lc.n)) / 256).astype(np.float32)
    c = sg.Code.from_linear_code(lc)
    out = sg.sogrand_decode(c, torch.from_numpy(x).cuda(), L=2, query_cap=2000, thr=thr)
    torch.cuda.synchronize()
    c.close()
    ref = oracle_lib.siso_batch(oracle_lib.OracleCode(lc), x, L=2, cap=2000, thr=float(np.float32(thr)))
    assert (ref["queries"] == 1).all() == (thr > 1e-38)
    np.testing.assert_array_equal(out["queries"].cpu().numpy(), ref["queries"])
    np.testing.assert_array_equal(out["list_count"].cpu().numpy(), ref["list_count"])


@pytest.mark.parametrize("thr", [1e-11, 1e-13])
def test_rule_with_64_bit_syndromes(env, oracle_lib, thr):
    """40 checks (7 of them independent, so that lists fill): the rule is asked
    at every listed word and the search goes on from the middle of a chunk of
    16-byte entries."""
    torch, sg = env
    base = ebch("ebch_64_57")
    rng = np.random.default_rng(6)
    H = np.concatenate([base.H, (rng.integers(0, 2, (33, 7)) @ base.H % 2).astype(np.uint8)])
    lc = LinearCode("ebch_64_57_40_checks", 64, 24, base.G, H)
    x = rng.standard_normal((60, 64)) * rng.choice([0.5, 2.0, 6.0], (60, 1)) + rng.choice([-3.0, 0.0, 3.0], (60, 1))
    x = x.astype(np.float32)
    c = sg.Code.from_linear_code(lc)
    out = sg.sogrand_decode(c, torch.from_numpy(x).cuda(), L=8, query_cap=3000, thr=thr)
    torch.cuda.synchronize()
    c.close()
    ref = oracle_lib.siso_batch(oracle_lib.OracleCode(lc), x, L=8, cap=3000, thr=float(np.float32(thr)))
    assert ref["list_count"].max() == 8
    compare_siso(lc, out, ref, f"40 checks thr={thr}")
