"""GPU parity of the numeric pass for rows whose products fit a block's
registers (129 to 8192 products by default), at the edges of its blocks and
bitmaps: rows of exactly 128 * 2^k products and one more, rows over one and
over several column windows (with empty windows between), rows whose products
all meet in one column or all stay apart, more nonzeros of A than threads, rows
of B that are empty."""
import numpy as np
import pytest

from paper_2112_10037_gb300 import gen
from parity import RTOL_F32, assert_structure_equal, assert_values_close, oracle_with_scale

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

EDGES = [129, 511, 512, 513, 1023, 1024, 1025, 2047, 2048, 2049, 4096, 4097, 8191, 8192, 8193]


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2112_10037_gb300 import build
    build.build()
    from paper_2112_10037_gb300 import api as a
    return a


def _operands(ncols, shape, seed):
    """A with one row per product count of EDGES; B's rows have 64 columns
    (rows 0..127), one column (the next 66) or none (the rest).  `shape`: where
    B's columns lie."""
    rng = np.random.default_rng(seed)
    wide, single, empty = 128, 66, 9000
    cols = []
    for k in range(wide):
        if shape == "spread":
            c = rng.choice(ncols, 64, replace=False)
        elif shape == "meet":  # every long row of B holds the same columns
            c = np.linspace(0, ncols - 1, 64).astype(np.int64)
        else:  # two clusters at both ends
            c = np.concatenate([rng.choice(80, 32, replace=False), ncols - 1 - rng.choice(80, 32, replace=False)])
        cols.append(np.sort(c))
    for k in range(single):
        cols.append(np.array([rng.integers(ncols) if shape != "meet" else 7]))
    counts = np.concatenate([np.full(wide, 64), np.ones(single, np.int64), np.zeros(empty, np.int64)])
    rp = np.concatenate([[0], np.cumsum(counts)]).astype(np.int32)
    ci = np.concatenate(cols).astype(np.int32)
    B = gen.CSR(len(counts), ncols, rp, ci, rng.standard_normal(len(ci))).check()
    rows = []
    for i, p in enumerate(EDGES):
        ones = p % 64 if p < 8192 else p - 127 * 64  # 8192, 8193: 127 long rows and 64 or more single ones
        longs = (p - ones) // 64
        ks = np.concatenate([rng.choice(wide, longs, replace=False), wide + np.arange(ones)])
        if i % 3 == 0:  # many nonzeros of A that reach nothing
            ks = np.concatenate([ks, wide + single + rng.choice(empty, 2500, replace=False)])
        rows.append(np.sort(ks))
    arp = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int32)
    aci = np.concatenate(rows).astype(np.int32)
    A = gen.CSR(len(rows), B.nrows, arp, aci, rng.standard_normal(len(aci))).check()
    return A, B


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("ncols,shape", [(300, "spread"), (5000, "meet"), (70001, "spread"), (600_000, "spread"),
                                         (600_000, "ends"), (3_000_000, "ends")])
def test_block_and_window_edges(api, oracle_mod, dtype, ncols, shape):
    A, B = _operands(ncols, shape, 5)
    dA = api.DeviceCSR.from_host(A, dtype=dtype)
    dB = api.DeviceCSR.from_host(B, dtype=dtype)
    got = api.spgemm(dA, dB).to_host()
    if dtype == torch.float32:
        A, B = (M.astype(np.float32).astype(np.float64) for M in (A, B))
    R, S = oracle_with_scale(oracle_mod, A, B)
    assert_structure_equal(got, R)
    assert_values_close(got.vals, R.vals, S, *([RTOL_F32] if dtype == torch.float32 else []))


@pytest.mark.parametrize("semiring", ["min_plus", "max_plus", "or_and"])
@pytest.mark.parametrize("ncols,shape", [(300, "spread"), (600_000, "ends")])
def test_semirings(api, oracle_mod, semiring, ncols, shape):
    A, B = _operands(ncols, shape, 6)
    got = api.spgemm_semiring(api.DeviceCSR.from_host(A), api.DeviceCSR.from_host(B), semiring).to_host()
    R = oracle_mod.spgemm(A, B)
    assert_structure_equal(got, R)
    assert np.array_equal(got.vals, oracle_mod.masked_semiring(A, B, R, semiring))


def test_infinities_and_nan(api, oracle_mod):
    """Special values reach exactly the entries the oracle gives them."""
    A, B = _operands(5000, "meet", 7)
    A.vals[::37], A.vals[5::91], B.vals[3::113] = np.inf, np.nan, -np.inf
    got = api.spgemm(api.DeviceCSR.from_host(A), api.DeviceCSR.from_host(B)).to_host()
    R = oracle_mod.spgemm(A, B)
    assert_structure_equal(got, R)
    assert np.array_equal(np.isnan(got.vals), np.isnan(R.vals))
    inf = np.isinf(R.vals)
    assert np.array_equal(got.vals[inf], R.vals[inf]) and np.array_equal(np.isinf(got.vals), inf)


@pytest.mark.parametrize("ncols", [9000, 200_000])
@pytest.mark.parametrize("num_block_min", [256, 4096])
def test_block_window_before_the_registers(api, oracle_mod, ncols, num_block_min):
    """Rows of at most 8192 products that the block window takes by an option:
    its run lists of B are built although no row is longer."""
    A, B = _operands(ncols, "spread", 8)
    keep = np.flatnonzero(np.array(EDGES) <= 8192)
    A = oracle_mod.select_rows(A, keep)
    got = api.spgemm(api.DeviceCSR.from_host(A), api.DeviceCSR.from_host(B), num_block_min=num_block_min).to_host()
    R, S = oracle_with_scale(oracle_mod, A, B)
    assert_structure_equal(got, R)
    assert_values_close(got.vals, R.vals, S)


@pytest.mark.parametrize("ncols", [5000, 70001])
def test_unsorted_rows_of_b_are_reported(api, oracle_mod, ncols):
    """Rows of B whose last column is their second smallest (the span that the
    analysis takes from their ends is too narrow), not validated: an error, and
    nothing outside the blocks' bitmaps."""
    from paper_2112_10037_gb300 import _native as nat
    A, B = _operands(ncols, "spread", 9)
    A = oracle_mod.select_rows(A, np.flatnonzero(np.array(EDGES) <= 2048))
    for k in range(128):
        s, e = B.row_ptr[k], B.row_ptr[k + 1]
        B.col_idx[s + 1:e] = B.col_idx[s + 1:e][::-1].copy()
    dA, dB = api.DeviceCSR.from_host(A), api.DeviceCSR.from_host(B)
    with pytest.raises(nat.SpgemmError) as e:
        plan = api.Plan(dA, dB)
        plan.symbolic()
        plan.numeric(dA.vals, dB.vals)
        plan.check()
    assert nat.STATUS_NAMES[e.value.status] == "SPGEMM_ERR_UNSORTED_INPUT"


@pytest.mark.parametrize("width", [9, 30, 60, 100, 250, 500, 1000, 2000])
@pytest.mark.parametrize("nrows", [40, 30_000])
def test_fp32_products_that_meet_are_fused(api, nrows, width):
    """Every column is x*y and -x*y: the first is rounded, the second fused, so
    what is left is exactly the first one's rounding error, with either sign (a
    rounded second product would leave 0).  Warp tables, lanes (many rows),
    block registers."""
    if nrows * width > 1_000_000:
        nrows = 500
    rng = np.random.default_rng(width)
    x, y = (rng.uniform(1, 2, n).astype(np.float32) for n in (nrows, width))
    cols = np.sort(rng.choice(70_001, width, replace=False)).astype(np.int32)
    B = gen.CSR(2, 70_001, np.array([0, width, 2 * width], np.int32), np.tile(cols, 2), np.tile(y, 2).astype(np.float64))
    A = gen.CSR(nrows, 2, (2 * np.arange(nrows + 1)).astype(np.int32), np.tile(np.array([0, 1], np.int32), nrows),
                np.stack([x, -x], 1).ravel().astype(np.float64))
    got = api.spgemm(*(api.DeviceCSR.from_host(M, dtype=torch.float32) for M in (A, B))).to_host()
    err = (x[:, None] * y).astype(np.float64) - x[:, None].astype(np.float64) * y
    assert np.count_nonzero(err) > 0.9 * err.size
    assert np.array_equal(np.abs(got.vals.reshape(nrows, width).astype(np.float64)), np.abs(err))


def test_fp32_infinities_and_nan(api, oracle_mod):
    """The same for FP32, whose products are fused by compare-and-swap."""
    A, B = _operands(5000, "meet", 7)
    A.vals[::37], A.vals[5::91], B.vals[3::113] = np.inf, np.nan, -np.inf
    got = api.spgemm(*(api.DeviceCSR.from_host(M, dtype=torch.float32) for M in (A, B))).to_host()
    R = oracle_mod.spgemm(A, B)
    assert_structure_equal(got, R)
    assert np.array_equal(np.isnan(got.vals), np.isnan(R.vals))
    inf = np.isinf(R.vals)
    assert np.array_equal(got.vals[inf], R.vals[inf]) and np.array_equal(np.isinf(got.vals), inf)
