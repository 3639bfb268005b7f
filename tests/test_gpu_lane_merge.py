"""GPU parity of the lane-per-row merge (rows of at most 8 nonzeros of A and
64 products): one to eight B rows of uneven and zero length, 1 to 64 outputs
(the collected groups of 8 full, ragged and empty), columns that all meet or
all stay apart, a last warp of few rows; the same rows beside one row of 9
nonzeros; and both in numbers below and above those that take a lane per row
(fewer take a warp each)."""
import numpy as np
import pytest

from paper_2112_10037_gb300 import gen
from parity import RTOL_F32, assert_structure_equal, assert_values_close, oracle_with_scale

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2112_10037_gb300 import build
    build.build()
    from paper_2112_10037_gb300 import api as a
    return a


def _operands(ncols, nine, nrows=1003, seed=3):
    rng = np.random.default_rng(seed)
    blen = np.minimum(np.repeat([0, 1, 2, 7, 8, 9, 16, 31, 64], 40), ncols)
    B = gen.random_rows(len(blen), ncols, blen, rng)
    rows = []
    for i in range(nrows):
        n = 1 + i % 8
        ks = np.sort(rng.choice(len(blen), n, replace=False))
        while blen[ks].sum() > 64:
            ks = ks[:-1] if len(ks) > 1 else np.array([45])
        rows.append(ks)
    if nine:
        rows[500] = np.arange(40, 49)
    rp = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int32)
    ci = np.concatenate(rows).astype(np.int32)
    return gen.CSR(len(rows), len(blen), rp, ci, rng.standard_normal(len(ci))).check(), B


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("ncols", [64, 100_000])
@pytest.mark.parametrize("nine", [False, True])
@pytest.mark.parametrize("nrows", [1003, 50_003, 320_003])
def test_rows(api, oracle_mod, nrows, ncols, nine, dtype):
    A, B = _operands(ncols, nine, nrows)
    got = api.spgemm(api.DeviceCSR.from_host(A, dtype=dtype), api.DeviceCSR.from_host(B, dtype=dtype)).to_host()
    if dtype == torch.float32:
        A, B = (M.astype(np.float32).astype(np.float64) for M in (A, B))
    R, S = oracle_with_scale(oracle_mod, A, B)
    assert_structure_equal(got, R)
    assert_values_close(got.vals, R.vals, S, *([RTOL_F32] if dtype == torch.float32 else []))


@pytest.mark.parametrize("semiring", ["min_plus", "max_plus", "or_and"])
@pytest.mark.parametrize("nrows,nine", [(1003, False), (50_003, False), (320_003, True)])
def test_semirings(api, oracle_mod, nrows, nine, semiring):
    A, B = _operands(64, nine, nrows)
    got = api.spgemm_semiring(api.DeviceCSR.from_host(A), api.DeviceCSR.from_host(B), semiring).to_host()
    R = oracle_mod.spgemm(A, B)
    assert_structure_equal(got, R)
    assert np.array_equal(got.vals, oracle_mod.masked_semiring(A, B, R, semiring))
