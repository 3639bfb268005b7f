"""GPU parity of the adjoint where its kernels hand over to each other: rows of
C at the edges of what a block stages in shared memory (128 and 4096 entries,
one bitmap of columns), rows of B of average length below and above the lane
groups' sizes, columns of A with more terms than a lane's chain takes, one
gradient at a time, and calls on two streams, named by two handles or by one
(the per-thread stream's)."""
import threading

import numpy as np
import pytest

from paper_2112_10037_gb300 import gen
from parity import abs_csr, max_rel_err

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


def _edge_operands(ncols, blen, seed):
    """A's rows reach 0, 1, 127..130, 1000 and 4094..4098 distinct columns:
    B's rows are disjoint runs of `blen` columns, and single columns after
    them; every row of A also holds column 0 of B's rows (a hub: one long
    column sum)."""
    rng = np.random.default_rng(seed)
    runs = 4200 // blen
    step = ncols // (runs * blen + 64)
    place = np.arange(runs * blen + 64, dtype=np.int64) * step + step // 2
    lens = np.concatenate([np.full(runs, blen), np.ones(64, np.int64), [0]])
    rp = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    order = rng.permutation(runs * blen)  # runs interleave over the whole width
    ci = np.concatenate([np.sort(place[order[k * blen:(k + 1) * blen]]) for k in range(runs)] + [place[runs * blen:]])
    B = gen.CSR(len(lens), ncols, rp, ci.astype(np.int32), rng.standard_normal(len(ci))).check()
    rows = []
    for want in [0, 1, 127, 128, 129, 130, 1000, 4094, 4095, 4096, 4097, 4098] + [blen] * 700:
        n = min(want // blen, runs)
        ones = min(want - n * blen, 64)
        ks = np.concatenate([np.arange(n), runs + np.arange(ones), [len(lens) - 1] if want % 2 else []])
        rows.append(np.sort(ks).astype(np.int64))
    arp = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int32)
    aci = np.concatenate(rows).astype(np.int32)
    return gen.CSR(len(rows), B.nrows, arp, aci, rng.standard_normal(len(aci))).check(), B


def _reference(oracle_mod, A, B, W):
    C = oracle_mod.spgemm(A, B)
    da, db = oracle_mod.backward(A, B, C.row_ptr, C.col_idx, W)
    sa, sb = oracle_mod.backward(abs_csr(A), abs_csr(B), C.row_ptr, C.col_idx, np.abs(W))
    return da, db, sa, sb


@pytest.mark.parametrize("dtype,tol", [(torch.float64, 1e-12), (torch.float32, 2e-4)])
@pytest.mark.parametrize("ncols", [5000, 600_000])
@pytest.mark.parametrize("blen", [7, 15, 60])
def test_row_edges(api, oracle_mod, blen, ncols, dtype, tol):
    A, B = _edge_operands(ncols, blen, blen)
    dA, dB = api.DeviceCSR.from_host(A, dtype=dtype), api.DeviceCSR.from_host(B, dtype=dtype)
    plan = api.Plan(dA, dB, dtype=dtype, backward=True)
    _, nnz = plan.symbolic()
    plan.numeric(dA.vals, dB.vals)
    W = np.random.default_rng(1).standard_normal(nnz).astype(np.float32).astype(np.float64)
    dW = torch.from_numpy(W).to(device="cuda", dtype=dtype)
    da, db = plan.backward(dA.vals, dB.vals, dW)
    only_a, none_b = plan.backward(dA.vals, dB.vals, dW, need_b=False)
    none_a, only_b = plan.backward(dA.vals, dB.vals, dW, need_a=False)
    torch.cuda.synchronize()
    plan.check()
    assert none_a is None and none_b is None
    assert torch.equal(da, only_a) and torch.equal(db, only_b)
    if dtype == torch.float32:
        A, B = (M.astype(np.float32).astype(np.float64) for M in (A, B))
    ra, rb, sa, sb = _reference(oracle_mod, A, B, W)
    assert max_rel_err(da.double().cpu().numpy(), ra, sa) <= tol
    assert max_rel_err(db.double().cpu().numpy(), rb, sb) <= tol
    plan.close()


def test_two_streams(api):
    """Calls on one plan from two streams give what each gives alone."""
    A = gen.random_rows(3000, 3000, np.full(3000, 40), np.random.default_rng(3))
    dA = api.DeviceCSR.from_host(A)
    plan = api.Plan(dA, dA, backward=True)
    _, nnz = plan.symbolic()
    plan.numeric(dA.vals, dA.vals)
    gen_ = torch.Generator(device="cuda").manual_seed(1)
    ws = [torch.randn(nnz, generator=gen_, device="cuda", dtype=torch.float64) for _ in range(2)]
    alone = [plan.backward(dA.vals, dA.vals, w) for w in ws]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in ws]
    home = plan.stream
    got = []
    for _ in range(5):
        for s, w in zip(streams, ws):
            plan.stream = int(s.cuda_stream)
            with torch.cuda.stream(s):
                got.append(plan.backward(dA.vals, dA.vals, w))
    torch.cuda.synchronize()
    plan.stream = home
    for i, (da, db) in enumerate(got):
        assert torch.equal(da, alone[i % 2][0]) and torch.equal(db, alone[i % 2][1])
    plan.close()


def _staged_operands(ncols, blen, seed):
    """Every row of A reaches 127..130, 1000 or 4094..4098 distinct columns or
    none, from rows of B of `blen` columns; products enough for staged rows."""
    rng = np.random.default_rng(seed)
    runs = 4200 // blen
    place = np.sort(rng.choice(ncols, runs * blen + 64, replace=False))
    order = rng.permutation(runs * blen)
    lens = np.concatenate([np.full(runs, blen), np.ones(64, np.int64), [0]])
    rp = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    ci = np.concatenate([np.sort(place[order[k * blen:(k + 1) * blen]]) for k in range(runs)] + [place[runs * blen:]])
    # `blen` columns in a row of B, 64 rows of one more: an average near blen
    B = gen.CSR(len(lens), ncols, rp, ci.astype(np.int32), rng.standard_normal(len(ci))).check()
    rows = []
    for want in [127, 128, 129, 130, 1000, 0] + [4094, 4095, 4096, 4097, 4098, 2000, 2500] * 6:
        n = min(want // blen, runs)
        ks = np.concatenate([rng.choice(runs, n, replace=False), runs + np.arange(min(want - n * blen, 64))])
        rows.append(np.sort(ks).astype(np.int64))
    arp = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int32)
    aci = np.concatenate(rows).astype(np.int32)
    return gen.CSR(len(rows), B.nrows, arp, aci, rng.standard_normal(len(aci))).check(), B


def _run(api, A, B, dtype, **want):
    """(dA, dB, launches of the call, dC) of one plan."""
    from paper_2112_10037_gb300 import _native as nat
    dA, dB = api.DeviceCSR.from_host(A, dtype=dtype), api.DeviceCSR.from_host(B, dtype=dtype)
    plan = api.Plan(dA, dB, dtype=dtype, backward=True)
    _, nnz = plan.symbolic()
    plan.numeric(dA.vals, dB.vals)
    W = np.random.default_rng(1).standard_normal(nnz).astype(np.float32).astype(np.float64)
    before = nat.spgemm_plan_launches(plan.handle)
    da, db = plan.backward(dA.vals, dB.vals, torch.from_numpy(W).to(device="cuda", dtype=dtype), **want)
    n = nat.spgemm_plan_launches(plan.handle) - before
    torch.cuda.synchronize()
    plan.check()
    plan.close()
    return da, db, n, W


@pytest.mark.parametrize("dtype,tol", [(torch.float64, 1e-12), (torch.float32, 2e-4)])
@pytest.mark.parametrize("ncols", [5000, 100_000])
@pytest.mark.parametrize("blen", [9, 16, 60])
def test_staged_rows(api, oracle_mod, blen, ncols, dtype, tol):
    A, B = _staged_operands(ncols, blen, blen)
    da, db, n, W = _run(api, A, B, dtype)
    assert n == 3  # staged rows, the other rows, the columns
    only_a, _, _, _ = _run(api, A, B, dtype, need_b=False)
    _, only_b, _, _ = _run(api, A, B, dtype, need_a=False)
    assert torch.equal(da, only_a) and torch.equal(db, only_b)
    if dtype == torch.float32:
        A, B = (M.astype(np.float32).astype(np.float64) for M in (A, B))
    ra, rb, sa, sb = _reference(oracle_mod, A, B, W)
    assert max_rel_err(da.double().cpu().numpy(), ra, sa) <= tol
    assert max_rel_err(db.double().cpu().numpy(), rb, sb) <= tol


@pytest.mark.parametrize("kind", ["stencil", "power", "short", "band"])
def test_searched_rows(api, oracle_mod, kind):
    """Products that staged rows or a buffer in chunks would slow down: a stencil
    of three chunks and a band of two (a search per term of each gradient), a
    power-law graph and uniform rows of few products (one search for both, then
    the columns).  dA alone is one launch, and the same bits."""
    rng = np.random.default_rng(2)
    if kind == "stencil":
        A = gen.laplacian_3d(80)
    elif kind == "power":
        A = gen.rmat(11, 16, seed=3)
    elif kind == "band":
        cols = np.arange(9000)[:, None] + np.arange(-16, 17)[None, :]
        ok = (cols >= 0) & (cols < 9000)
        A = gen.CSR(9000, 9000, np.concatenate([[0], np.cumsum(ok.sum(1))]).astype(np.int32),
                    cols[ok].astype(np.int32), rng.standard_normal(int(ok.sum()))).check()
    else:
        A = gen.random_rows(20000, 20000, rng.integers(6, 13, 20000), rng)
    da, db, n, W = _run(api, A, A, torch.float64)
    assert n == 2
    only_a, _, n, _ = _run(api, A, A, torch.float64, need_b=False)
    assert n == 1 and torch.equal(da, only_a)
    ra, rb, sa, sb = _reference(oracle_mod, A, A, W)
    assert max_rel_err(da.cpu().numpy(), ra, sa) <= 1e-12
    assert max_rel_err(db.cpu().numpy(), rb, sb) <= 1e-12


# (4500, 4000): 18 M products, more than one chunk of the buffer
@pytest.mark.parametrize("terms,width", [(129, 64), (256, 64), (512, 64), (4096, 300), (4500, 4000)])
def test_long_sums_keep_their_chains(api, terms, width):
    """dB's sums of more than 128 terms are 32 chains of every 32nd term and a
    tree of five levels.  A = one column, B = one row, positive FP32 operands:
    a rounding is u/sqrt(3) of its partial sum in the root mean square (u =
    2^-24); the m = terms/32 of a chain, whose partial sums grow evenly, come to
    sqrt(m/3) of the chain's sum, over 32 chains sqrt(m/96) of the whole, the
    tree's levels to 1, 1/2, ... of it, squared: less than 2.  1.3 for the
    sample.  (One chain of 256
    terms comes to sqrt(256/3), six times the bound.)"""
    rng = np.random.default_rng(terms)
    arp = np.arange(terms + 1, dtype=np.int32)
    A = gen.CSR(terms, 1, arp, np.zeros(terms, np.int32), rng.uniform(0.5, 1.5, terms).astype(np.float32))
    B = gen.CSR(1, width, np.array([0, width], np.int32), np.arange(width, dtype=np.int32),
                rng.uniform(0.5, 1.5, width).astype(np.float32))
    dA, dB = (api.DeviceCSR.from_host(M, dtype=torch.float32) for M in (A, B))
    plan = api.Plan(dA, dB, dtype=torch.float32, backward=True)
    _, nnz = plan.symbolic()
    plan.numeric(dA.vals, dB.vals)
    W = rng.uniform(0.5, 1.5, nnz).astype(np.float32)
    _, db = plan.backward(dA.vals, dB.vals, torch.from_numpy(W).cuda())
    torch.cuda.synchronize()
    plan.check()
    plan.close()
    ref = A.vals.astype(np.float64) @ W.reshape(terms, width).astype(np.float64)
    err = np.sqrt(np.mean(((db.double().cpu().numpy() - ref) / ref) ** 2))
    bound = 1.3 * 2.0 ** -24 / np.sqrt(3.0) * np.sqrt(-(-terms // 32) / 96.0 + 2.0)
    assert err <= bound


def test_per_thread_streams(api):
    """Two host threads that both name the per-thread stream: one handle, a
    different stream in each thread, one product buffer."""
    from paper_2112_10037_gb300 import _native as nat
    A = gen.random_rows(3000, 3000, np.full(3000, 40), np.random.default_rng(3))
    dA = api.DeviceCSR.from_host(A)
    plan = api.Plan(dA, dA, backward=True)
    _, nnz = plan.symbolic()
    plan.numeric(dA.vals, dA.vals)
    gen_ = torch.Generator(device="cuda").manual_seed(1)
    ws = [torch.randn(nnz, generator=gen_, device="cuda", dtype=torch.float64) for _ in range(2)]
    alone = [plan.backward(dA.vals, dA.vals, w) for w in ws]
    reps = 8
    out = [[(torch.zeros_like(dA.vals), torch.zeros_like(dA.vals)) for _ in range(reps)] for _ in ws]
    torch.cuda.synchronize()
    start, failed = threading.Barrier(2), []

    def work(i):
        try:
            torch.cuda.set_device(0)
            start.wait()
            for da, db in out[i]:
                nat.spgemm_backward(plan.handle, dA.vals.data_ptr(), dA.vals.data_ptr(), plan.row_ptr.data_ptr(),
                                    plan.col_idx.data_ptr(), ws[i].data_ptr(), da.data_ptr(), db.data_ptr(),
                                    2)  # cudaStreamPerThread
        except Exception as e:  # reported by the main thread
            failed.append(e)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not failed
    for i, pairs in enumerate(out):
        for da, db in pairs:
            assert torch.equal(da, alone[i][0]) and torch.equal(db, alone[i][1])
    plan.close()


@pytest.mark.parametrize("kind,dtype", [("staged", torch.float64), ("chunks", torch.float32), ("long", torch.float64)])
def test_captured_calls_run_beside_others(api, kind, dtype):
    """Two graphs captured from one plan's adjoint and eager calls, all at once
    on three streams: the bits of an eager call alone.  Rows staged in shared
    memory, two chunks of the buffer, sums of more than 128 terms."""
    from paper_2112_10037_gb300 import _native as nat
    rng = np.random.default_rng(5)
    if kind == "staged":
        A = gen.random_rows(3000, 3000, np.full(3000, 40), rng)
    elif kind == "chunks":
        A = gen.random_rows(20000, 20000, np.full(20000, 32), rng)
    else:
        A = gen.random_rows(2000, 90, rng.integers(2, 20, 2000), rng)
    B = gen.random_rows(90, 4000, np.full(90, 60), rng) if kind == "long" else A
    dA, dB = api.DeviceCSR.from_host(A, dtype=dtype), api.DeviceCSR.from_host(B, dtype=dtype)
    plan = api.Plan(dA, dB, dtype=dtype, backward=True)
    _, nnz = plan.symbolic()
    plan.numeric(dA.vals, dB.vals)
    gen_ = torch.Generator(device="cuda").manual_seed(1)
    ws = [torch.randn(nnz, generator=gen_, device="cuda", dtype=dtype) for _ in range(3)]
    alone = [plan.backward(dA.vals, dB.vals, w) for w in ws]
    outs = [(torch.zeros_like(dA.vals), torch.zeros_like(dB.vals)) for _ in ws]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in ws]

    def call(i):
        nat.spgemm_backward(plan.handle, dA.vals.data_ptr(), dB.vals.data_ptr(), plan.row_ptr.data_ptr(),
                            plan.col_idx.data_ptr(), ws[i].data_ptr(), outs[i][0].data_ptr(), outs[i][1].data_ptr(),
                            int(streams[i].cuda_stream))

    graphs = []
    for i in range(2):
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=streams[i]):
            call(i)
        graphs.append(g)
    for _ in range(10):
        for i in range(2):
            with torch.cuda.stream(streams[i]):
                graphs[i].replay()
        call(2)
    torch.cuda.synchronize()
    plan.check()
    for (da, db), (ra, rb) in zip(outs, alone):
        assert torch.equal(da, ra) and torch.equal(db, rb)
    plan.close()
