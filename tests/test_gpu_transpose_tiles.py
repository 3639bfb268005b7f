"""GPU transpose where its tiles end: matrices whose digits take tiles of 2048
and of 4096 entries, with entry counts just below, at and above one and several
tiles, with and without source positions."""
import numpy as np
import pytest

from paper_2112_10037_gb300 import gen

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


# columns: 7 bits in one pass, 2 x 5, 2 x 7 (small tiles); 9, 2 x 8, 2 x 9 (large)
@pytest.mark.parametrize("ncols", [128, 600, 16384, 512, 65536, 262144])
@pytest.mark.parametrize("nnz", [2047, 2048, 2049, 4095, 4096, 4097, 20481])
def test_tile_edges(api, ncols, nnz):
    rng = np.random.default_rng(nnz)
    nrows = 400
    lens = np.full(nrows, nnz // nrows)
    lens[: nnz - lens.sum()] += 1
    M = gen.random_rows(nrows, ncols, lens, rng, values="int")
    dM = api.DeviceCSR.from_host(M)
    order = np.argsort(M.col_idx, kind="stable")
    rows = np.repeat(np.arange(nrows), np.diff(M.row_ptr))[order]
    rp = np.concatenate([[0], np.cumsum(np.bincount(M.col_idx, minlength=ncols))])
    for want_src in (False, True):
        got = api.transpose(dM, want_src=want_src)
        T, src = got if want_src else (got, None)
        assert np.array_equal(T.row_ptr.cpu().numpy(), rp)
        assert np.array_equal(T.col_idx.cpu().numpy(), rows)
        assert np.array_equal(T.vals.cpu().numpy(), M.vals[order])
        if want_src:
            assert np.array_equal(src.cpu().numpy(), order)


def test_columns_out_of_range_leave_empty_rows(api):
    """Every other entry's column is out of range: an error, and a row pointer
    of an empty matrix (every step down of the columns would fill rows)."""
    from paper_2112_10037_gb300 import _native as nat
    n, nnz = 10_000, 3000
    rp = torch.tensor([0, nnz], dtype=torch.int32, device="cuda")
    ci = torch.arange(nnz, dtype=torch.int32, device="cuda")
    ci[1::2] += 3 << 16
    t_rp = torch.full((n + 1,), -1, dtype=torch.int32, device="cuda")
    t_ci = torch.zeros(nnz, dtype=torch.int32, device="cuda")
    M = api.DeviceCSR(1, n, rp, ci, torch.ones(nnz, dtype=torch.float64, device="cuda")).c_struct()
    size = nat.spgemm_transpose_workspace_size(1, n, nnz)
    ws = torch.empty(size, dtype=torch.uint8, device="cuda")
    s = int(torch.cuda.current_stream().cuda_stream)
    nat.spgemm_transpose(M, 0, t_rp.data_ptr(), t_ci.data_ptr(), 0, 0, ws.data_ptr(), size, s)
    with pytest.raises(nat.SpgemmError) as e:
        nat.spgemm_transpose_check(ws.data_ptr(), s)
    assert nat.STATUS_NAMES[e.value.status] == "SPGEMM_ERR_UNSORTED_INPUT"
    assert not t_rp.any()


# rows walked from entry to entry (below 16 rows per entry and tile), searched
# per entry (above), and both in one matrix
@pytest.mark.parametrize("nrows,nnz", [(32_000, 2048), (40_000, 2048), (3_000_000, 1), (3_000_000, 2), (3_000_000, 5001),
                                       (70_000, 4097)])
@pytest.mark.parametrize("ncols", [600, 65536])
def test_far_more_rows_than_entries(api, nrows, nnz, ncols):
    rng = np.random.default_rng(nnz)
    lens = np.zeros(nrows, np.int64)
    at = np.concatenate([[0, nrows - 1], rng.integers(0, nrows, max(0, nnz - 2))])[:nnz]  # both ends
    np.add.at(lens, at[: nnz // 2], 1)
    np.add.at(lens, at[nnz // 2:] // 50, 1)  # half of them among the first rows
    M = gen.random_rows(nrows, ncols, np.minimum(lens, ncols), rng, values="int")
    T = api.transpose(api.DeviceCSR.from_host(M))
    order = np.argsort(M.col_idx, kind="stable")
    assert np.array_equal(T.row_ptr.cpu().numpy(), np.concatenate([[0], np.cumsum(np.bincount(M.col_idx, minlength=ncols))]))
    assert np.array_equal(T.col_idx.cpu().numpy(), np.repeat(np.arange(nrows), np.diff(M.row_ptr))[order])
    assert np.array_equal(T.vals.cpu().numpy(), M.vals[order])
