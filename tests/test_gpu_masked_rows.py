"""GPU parity of the masked product where its ways of testing a product hand
over: mask rows at the edges of the staged columns (384) and of the hashed
bitmap (2048), parts of a row of A that form few and many products, rows of B
below, at and above a warp's width, rows of A over several 32-nonzero units."""
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


def _operands(seed):
    rng = np.random.default_rng(seed)
    blen = np.array([0, 1, 2, 31, 32, 33, 63, 127, 128, 129, 300, 5000] * 8)
    n = 9000
    B = gen.random_rows(len(blen), n, blen, rng, values="int")
    mlen = np.array([0, 1, 2, 31, 33, 383, 384, 385, 2047, 2048, 2049, 4100] * 6)
    M = gen.random_rows(len(mlen), n, mlen, rng, values="int")
    A = gen.random_rows(len(mlen), B.nrows, rng.choice([0, 1, 2, 3, 31, 32, 33, 70], len(mlen)), rng, values="int")
    return A, B, M


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("semiring", ["plus_times", "min_plus", "max_plus", "or_and"])
def test_edges(api, oracle_mod, semiring, dtype):
    A, B, M = _operands(4)  # whole numbers: every sum is exact in both types
    dA, dB, dM = (api.DeviceCSR.from_host(X, dtype=dtype) for X in (A, B, M))
    got = api.masked_semiring(dA, dB, dM, semiring).double().cpu().numpy()
    ref = (oracle_mod.masked(A, B, M, use_mask_values=False) if semiring == "plus_times"
           else oracle_mod.masked_semiring(A, B, M, semiring))
    assert np.array_equal(got, ref)


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("semiring", ["plus_times", "min_plus", "or_and"])
def test_rows_for_blocks(api, oracle_mod, semiring, dtype):
    """Rows of A at the edges of what blocks take (64 nonzeros, 4 mask columns
    each), over one and several units of 256, mask rows at the edges of the
    staged accumulators (1536) and columns (4608, 3072 in FP32), short rows
    between them."""
    rng = np.random.default_rng(8)
    blen = rng.choice([0, 1, 5, 31, 32, 33, 127, 129, 400], 1600)
    blen[[3, 300]] = 9000
    n = 12000
    B = gen.random_rows(len(blen), n, blen, rng, values="int")
    alen = np.array([63, 64, 64, 65, 3, 255, 256, 257, 0, 520, 700, 600, 64, 1, 100, 512, 513, 66, 1100, 1100,
                     1600, 1600] + [1600] * 5)
    mlen = np.array([252, 256, 257, 1, 40, 0, 1024, 1028, 5, 1535, 1536, 1537, 64, 9, 401, 2400, 2052, 264, 3072, 3073,
                     4608, 4609] + [3] * 5)
    A = gen.random_rows(len(alen), B.nrows, alen, rng, values="int")
    M = gen.random_rows(len(mlen), n, mlen, rng, values="int")
    assert M.nnz <= 2 * A.nnz  # denser masks leave every row to the warps
    dA, dB, dM = (api.DeviceCSR.from_host(X, dtype=dtype) for X in (A, B, M))
    got = api.masked_semiring(dA, dB, dM, semiring).double().cpu().numpy()
    ref = (oracle_mod.masked(A, B, M, use_mask_values=False) if semiring == "plus_times"
           else oracle_mod.masked_semiring(A, B, M, semiring))
    assert np.array_equal(got, ref)
