"""GPU parity of the banded accumulator (long rows by default): rows whose
outputs fill one band exactly, fall just short of it and run over into the
next, rows of more nonzeros than a block's threads (cursors in global memory),
rows over several bitmap windows with empty windows between, columns that all
rows of B share, B rows shorter and longer than a warp."""
import numpy as np
import pytest

from paper_2112_10037_gb300 import gen
from parity import RTOL_F32, assert_structure_equal, assert_values_close, oracle_with_scale

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

CAP = {torch.float64: 5120, torch.float32: 8192}  # ranks per band


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2112_10037_gb300 import build
    build.build()
    from paper_2112_10037_gb300 import api as a
    return a


def _check(api, oracle_mod, A, B, dtype):
    from paper_2112_10037_gb300 import _native as nat
    dA, dB = api.DeviceCSR.from_host(A, dtype=dtype), api.DeviceCSR.from_host(B, dtype=dtype)
    plan = api.Plan(dA, dB, dtype=dtype)
    nat.spgemm_plan_set_profiling(plan.handle, True)
    rp, _ = plan.symbolic()
    ci, v = plan.numeric(dA.vals, dB.vals)
    torch.cuda.synchronize()
    plan.check()
    assert nat.spgemm_plan_kernel_times(plan.handle)["num_block"] > 0  # the long rows' timer
    plan.close()
    got = gen.CSR(A.nrows, B.ncols, rp.cpu().numpy(), ci.cpu().numpy(), v.double().cpu().numpy())
    if dtype == torch.float32:
        A, B = (M.astype(np.float32).astype(np.float64) for M in (A, B))
    R, S = oracle_with_scale(oracle_mod, A, B)
    assert_structure_equal(got, R)
    assert_values_close(got.vals, R.vals, S, *([RTOL_F32] if dtype == torch.float32 else []))


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("ncols", [70_000, 262_144, 700_000])
def test_band_edges(api, oracle_mod, ncols, dtype):
    """Row i of A reaches exactly want[i] distinct columns, each twice."""
    rng = np.random.default_rng(ncols)
    cap = CAP[dtype]
    want = [cap - 1, cap, cap + 1, 2 * cap, 2 * cap + 31, 3 * cap + 1, 4500]
    cols = np.sort(rng.choice(ncols, 3 * cap + 64, replace=False))
    lens, pieces = [], []
    for w in want:  # the first w columns in pieces of uneven length, then once more in others
        for seed_off in (0, 1):
            cuts = np.sort(rng.choice(np.arange(1, w), 40, replace=False))
            for p in np.split(cols[:w], cuts):
                lens.append(len(p))
                pieces.append(p)
    rp = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    B = gen.CSR(len(lens), ncols, rp, np.concatenate(pieces).astype(np.int32),
                rng.standard_normal(int(rp[-1]))).check()
    per = 2 * 41
    arp = (np.arange(len(want) + 1) * per).astype(np.int32)
    A = gen.CSR(len(want), B.nrows, arp, np.arange(per * len(want), dtype=np.int32),
                rng.standard_normal(per * len(want))).check()
    _check(api, oracle_mod, A, B, dtype)


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("ncols", [40_000, 1_200_000])
def test_many_nonzeros_and_shared_columns(api, oracle_mod, ncols, dtype):
    """Rows of 100 to 1500 nonzeros; B's rows hold 3 to 200 columns, half of
    them from a set of 300 that every row draws from."""
    rng = np.random.default_rng(9)
    k = 2000
    hubs = rng.choice(ncols, 300, replace=False)
    rows = [np.unique(np.concatenate([rng.choice(hubs, n // 2, replace=False), rng.integers(0, ncols, n - n // 2)]))
            for n in rng.choice([3, 20, 31, 32, 33, 64, 200], k)]
    rp = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int32)
    B = gen.CSR(k, ncols, rp, np.concatenate(rows).astype(np.int32), rng.standard_normal(int(rp[-1]))).check()
    A = gen.random_rows(24, k, rng.choice([100, 511, 512, 513, 1024, 1500], 24), rng)
    _check(api, oracle_mod, A, B, dtype)


@pytest.mark.parametrize("semiring", ["min_plus", "max_plus", "or_and"])
def test_semirings(api, oracle_mod, semiring):
    rng = np.random.default_rng(4)
    B = gen.random_rows(300, 90_000, rng.integers(1, 900, 300), rng, values="int")
    A = gen.random_rows(12, 300, rng.integers(20, 200, 12), rng, values="int")
    got = api.spgemm_semiring(api.DeviceCSR.from_host(A), api.DeviceCSR.from_host(B), semiring).to_host()
    R = oracle_mod.spgemm(A, B)
    assert_structure_equal(got, R)
    assert np.array_equal(got.vals, oracle_mod.masked_semiring(A, B, R, semiring))


def _block_rows(n, kind, rng):
    """At least 16 M products in rows that the windows take: a band that
    straddles windows, dense blocks, 3000 columns that all rows share (one row of
    more than 65,536 products among them), every 50th row short."""
    if kind == "band":
        cols = np.arange(n)[:, None] + np.arange(-20, 21)[None, :]
        rows = [c[(c >= 0) & (c < n)] for c in cols]
    elif kind == "blocks":
        rows = [i // 40 * 40 + np.arange(min(40, n - i // 40 * 40)) for i in range(n)]
    else:
        rows = [np.sort(rng.choice(3000, 70, replace=False)) for _ in range(n)]
        rows[7] = np.sort(rng.choice(n, 1500, replace=False))
    for i in range(0, n, 50):
        rows[i] = rows[i][:3]
    rp = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int32)
    ci = np.concatenate(rows).astype(np.int32)
    return gen.CSR(n, n, rp, ci, rng.standard_normal(len(ci))).check()


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("kind,n", [("band", 12_000), ("blocks", 12_001), ("shared", 9_000), ("band", 40_000)])
def test_dense_rows_take_windows(api, oracle_mod, kind, n, dtype):
    """Many rows of many products on few columns: the windows' lists are built
    with the symbolic pass; a plan of a range of the rows reads them, and ranks its
    columns while they do not exist."""
    from paper_2112_10037_gb300 import _native as nat
    A = _block_rows(n, kind, np.random.default_rng(n))
    assert oracle_mod.row_products(A, A).sum() >= 16_000_000
    dA = api.DeviceCSR.from_host(A, dtype=dtype)
    plan = api.Plan(dA, dA, dtype=dtype)
    early = plan.rows(0, n - 300)
    early_rp, _ = early.symbolic()
    first = early.numeric(dA.vals, dA.vals)  # before the lists exist
    before = nat.spgemm_plan_launches(plan.handle)
    rp, _ = plan.symbolic()
    assert nat.spgemm_plan_launches(plan.handle) - before >= 6  # two symbolic, a scan, the lists' three
    ci, v = plan.numeric(dA.vals, dA.vals)
    late = plan.rows(100, n)
    late_rp, _ = late.symbolic()
    got = [(first, early_rp, 0, n - 300), (early.numeric(dA.vals, dA.vals), early_rp, 0, n - 300),
           (late.numeric(dA.vals, dA.vals), late_rp, 100, n)]
    torch.cuda.synchronize()
    plan.check()
    for p in (early, late):
        p.check()
    if dtype == torch.float32:
        A = A.astype(np.float32).astype(np.float64)
    R, S = oracle_with_scale(oracle_mod, A, A)
    C = gen.CSR(n, n, rp.cpu().numpy(), ci.cpu().numpy(), v.double().cpu().numpy())
    assert_structure_equal(C, R)
    assert_values_close(C.vals, R.vals, S, *([RTOL_F32] if dtype == torch.float32 else []))
    for (pci, pv), r, a, b in got:
        s, e = R.row_ptr[a], R.row_ptr[b]
        assert np.array_equal(r.cpu().numpy(), R.row_ptr[a:b + 1] - s)
        assert np.array_equal(pci.cpu().numpy(), R.col_idx[s:e])
        assert np.all(np.abs(pv.double().cpu().numpy() - R.vals[s:e]) <=
                      (RTOL_F32 if dtype == torch.float32 else 1e-12) * S[s:e])
    for p in (early, late, plan):
        p.close()


@pytest.mark.parametrize("semiring", ["min_plus", "or_and"])
def test_dense_rows_semirings(api, oracle_mod, semiring):
    A = _block_rows(12_000, "blocks", np.random.default_rng(1))
    got = api.spgemm_semiring(api.DeviceCSR.from_host(A), api.DeviceCSR.from_host(A), semiring).to_host()
    R = oracle_mod.spgemm(A, A)
    assert_structure_equal(got, R)
    assert np.array_equal(got.vals, oracle_mod.masked_semiring(A, A, R, semiring))
