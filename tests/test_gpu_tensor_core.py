"""The tensor-core paths (dense sparse-matrix products, float32 gradient) where their operands, their workspace or the
host's state are not the ordinary ones: each compared with plain torch in 64 bits or with the same call on a fresh
workspace."""

import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
U = 2.0 ** -24


@pytest.fixture(scope="module")
def C():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1905_07931_gb300 import csrtrain
    csrtrain.lib()
    return csrtrain


def _gen(seed):
    return torch.Generator("cuda").manual_seed(seed)


def _weights(m, k, density, seed):
    g = _gen(seed)
    w = torch.randn(m, k, device="cuda", generator=g)
    return w * (torch.rand(m, k, device="cuda", generator=g) < density)


def _csr(C, dense, ws, transposed=False, capacity=None):
    w = C.CSR(*dense.shape, capacity=capacity, transposed=transposed)
    C.csr_from_dense(dense.contiguous(), w, ws)
    return w


def _bits(t):
    return t.view(torch.int32)


@pytest.mark.parametrize("m,k,n", [(777, 4000, 333), (1300, 5000, 99)])   # column tiles of 256 and 128, all shared
def test_product_after_a_wait_that_gave_up(C, m, k, n):
    """A kernel that gives up waiting leaves counters behind; the status is cleared, the next product is right."""
    ws = C.Workspace(m, k, n)
    dense = _weights(m, k, 0.3, m)
    w = _csr(C, dense, ws)
    x = torch.randn(k, n, device="cuda", generator=_gen(n))
    want, got = (torch.full((m, n), float("nan"), device="cuda") for _ in range(2))
    C.launch_count(reset=True)
    C.spmm_fwd(w, x, want, ws)
    assert C.launch_count() == 2, "a shape of the tensor-core path"
    words = ws.buf[256:].view(torch.int32)
    for stale in (1, 0x101, 7):
        words.fill_(stale)           # counters and scratch alike
        ws.clear_status()
        C.spmm_fwd(w, x, got, ws)
        assert torch.equal(_bits(got), _bits(want))
    assert ws.status()[0] == 0


FIRST_CALLS = """
import threading, torch
from paper_1905_07931_gb300 import csrtrain as C
N, m, n = 24, 512, 256
g = torch.Generator("cuda").manual_seed(1)
dy, x = (torch.randn(m, n, device="cuda", generator=g) for _ in range(2))
ws = [C.Workspace(m, m, n) for _ in range(N + 1)]
out = [torch.zeros(m, m, device="cuda") for _ in range(N + 1)]
torch.cuda.synchronize()
launches, gate = [None] * N, threading.Barrier(N)
def call(i):
    torch.cuda.set_device(0)
    gate.wait()
    C.weight_grad_dense(dy, x, out[i], ws[i], precision=0)
    launches[i] = C.launch_count()
threads = [threading.Thread(target=call, args=(i,)) for i in range(N)]
[t.start() for t in threads]
[t.join() for t in threads]
C.weight_grad_dense(dy, x, out[N], ws[N], precision=0)
torch.cuda.synchronize()
assert launches == [2] * N, launches      # the tensor-core path in every thread
assert all(torch.equal(o, out[N]) for o in out)
"""


def test_first_calls_of_many_threads(C):
    """A process whose first calls come from many threads at once takes the same path in all of them."""
    r = subprocess.run([sys.executable, "-c", FIRST_CALLS], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]


@pytest.mark.parametrize("n", [256, 333])
@pytest.mark.parametrize("how", ["reversed", "shuffled", "twice"])
def test_product_of_rows_in_any_order(C, n, how):
    """Rows whose columns don't ascend, or that hold an entry of one column twice, are added up as they are stored."""
    m, k = 700, 4000
    ws = C.Workspace(m, k, n)
    dense = _weights(m, k, 0.3, 5)
    w = _csr(C, dense, ws)
    x = torch.randn(k, n, device="cuda", generator=_gen(n))
    b, e = (int(v) for v in w.row_ptr[[37, 38]])
    if how == "twice":
        w.col_idx[b + 9] = w.col_idx[b + 8]
    else:
        perm = torch.arange(e - b - 1, -1, -1) if how == "reversed" else torch.randperm(e - b)
        w.col_idx[b:e] = w.col_idx[b:e][perm.cuda()]
        w.val[b:e] = w.val[b:e][perm.cuda()]
    full = torch.zeros(m, k, device="cuda", dtype=torch.float64)
    nnz = int(w.row_ptr[-1])
    rows = torch.repeat_interleave(torch.arange(m, device="cuda"), (w.row_ptr[1:] - w.row_ptr[:-1]).long())
    full.index_put_((rows, w.col_idx[:nnz].long()), w.val[:nnz].double(), accumulate=True)
    mag = torch.zeros_like(full).index_put_((rows, w.col_idx[:nnz].long()), w.val[:nnz].double().abs(),
                                            accumulate=True)
    y = torch.full((m, n), float("nan"), device="cuda")
    C.spmm_fwd(w, x, y, ws)
    lens = (w.row_ptr[1:] - w.row_ptr[:-1]).double()[:, None]
    assert bool(((y.double() - full @ x.double()).abs() <= (lens + 2) * U * (mag @ x.double().abs())).all())
    assert ws.status()[0] == 0


def _us(call, reps=5):
    for _ in range(2):
        call()
    best = float("inf")
    for _ in range(reps):
        a, b = torch.cuda.Event(True), torch.cuda.Event(True)
        a.record()
        call()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b) * 1e3)
    return best


def test_product_with_values_out_of_range_costs_a_sparse_product(C):
    """One NaN in X, one infinity in W, or large values all over: right, and at the price of gathering every entry
    (2.6 times the tensor cores' at 20%, measured) and not that of a serial sum per element (40 to 130 times)."""
    m = k = 4096
    n = 256
    ws = C.Workspace(m, k, n)
    dense = _weights(m, k, 0.2, 3)
    w = _csr(C, dense, ws)
    x = torch.randn(k, n, device="cuda", generator=_gen(4))
    y = torch.empty(m, n, device="cuda")
    plain = _us(lambda: C.spmm_fwd(w, x, y, ws))
    lens = (dense != 0).sum(1, keepdim=True).double()
    for what in ("nan", "large", "weight"):
        xb, wb = x.clone(), w
        if what == "nan":
            xb[7, 3] = float("nan")
        elif what == "large":
            xb[5::64, 3::64] *= 2.0 ** 62
        else:
            db = dense.clone()
            db[9, 11] = -2.0 ** 100
            wb = _csr(C, db, ws)
        assert _us(lambda: C.spmm_fwd(wb, xb, y, ws)) < 10 * plain, what
        full, xc = (db if what == "weight" else dense).double(), xb.double()
        if what == "nan":
            xc[7, 3] = 0
        ref, mag = full @ xc, full.abs() @ xc.abs()
        if what == "nan":
            hit = torch.zeros(m, n, dtype=torch.bool, device="cuda")
            hit[:, 3] = dense[:, 7] != 0
            assert torch.equal(y.isnan(), hit)
            y[hit], ref[hit] = 0, 0
        assert bool(((y.double() - ref).abs() <= (lens + 3) * U * mag).all()), what
    assert ws.status()[0] == 0


def test_product_beside_another_kernel(C):
    """While another stream's kernel holds most of the GPU the pairs of shared tiles are not resident together: each
    gives up its wait, whoever counts in last does its share, and the sums are the same."""
    m, k, n = 4096, 4096, 256
    ws = C.Workspace(m, k, n)
    w = _csr(C, _weights(m, k, 0.2, 8), ws)
    x = torch.randn(k, n, device="cuda", generator=_gen(9))
    want, got = torch.empty(m, n, device="cuda"), torch.empty(m, n, device="cuda")
    C.spmm_fwd(w, x, want, ws)
    side, blocks = torch.cuda.Stream(), 120
    out = torch.empty(blocks * 512, device="cuda")
    torch.cuda.synchronize()
    for iters in (1 << 15, 1 << 17):
        assert C.lib().csrt_fma_peak_run(out.data_ptr(), blocks, iters, None, side.cuda_stream) == 0
        for _ in range(5):
            got.fill_(float("nan"))
            C.spmm_fwd(w, x, got, ws)
            assert torch.equal(_bits(got), _bits(want))
        side.synchronize()
    assert ws.status()[0] == 0


def _uniform(seed, lo, hi, *shape):
    return 10.0 ** (lo + (hi - lo) * torch.rand(*shape, device="cuda", generator=_gen(seed)))


@pytest.mark.parametrize("m,k,n", [(4096, 4096, 256), (1025, 4000, 333), (1300, 5000, 99)])
@pytest.mark.parametrize("what", ["samples", "rows", "tiny"])
def test_product_of_any_range(C, m, k, n, what):
    """An element of Y is as exact as its own terms allow, whatever the magnitudes around them: samples of very
    different scale in one batch, rows whose entries span 15 decades and meet features of the inverse scale, values down
    to float32's least. Each within float32's summation bound for its terms."""
    ws = C.Workspace(m, k, n)
    dense, x = _weights(m, k, 0.2, 1), torch.randn(k, n, device="cuda", generator=_gen(2))
    dy = torch.randn(m, n, device="cuda", generator=_gen(3))
    if what == "samples":
        s = _uniform(4, -30, 0, 1, n)
        x, dy = x * s, dy * s
    elif what == "rows":
        s = _uniform(5, -15, 0, k)
        dense, x = dense * s, x / s[:, None] * 1e-8
    else:
        dense = dense * 2.0 ** -122    # down to 2^-149, 27 binades, with features of 2^25
        x, dy = x * 2.0 ** 25, dy * 2.0 ** 25
    w = _csr(C, dense, ws, transposed=True)
    y, dx = torch.full((m, n), float("nan"), device="cuda"), torch.full((k, n), float("nan"), device="cuda")
    C.launch_count(reset=True)
    C.spmm_fwd(w, x, y, ws)
    assert C.launch_count() == 2, "a shape of the tensor-core path"
    C.spmm_bwd_t(w, dy, dx, ws)
    d = dense.double()
    for got, a, b in ((y, d, x), (dx, d.T, dy)):
        terms = (a != 0).sum(1, keepdim=True).double()
        lim = (terms + 64) * U * (a.abs() @ b.double().abs()) + 2.0 ** -149
        assert bool(((got.double() - a @ b.double()).abs() <= lim).all())
    assert ws.status()[0] == 0


@pytest.mark.parametrize("m,n", [(4096, 256), (1300, 99)])
def test_product_with_one_feature(C, m, n):
    """Sums of one term: a feature of 1 returns W's entry, any other one rounding of the product and the parts that are
    left out (at most 2^-24 of it each)."""
    k = 4096
    ws = C.Workspace(m, k, n)
    dense = _weights(m, k, 0.3, 6)
    w = _csr(C, dense, ws)
    at = torch.randperm(k, generator=torch.Generator().manual_seed(1))[:n].cuda()
    x = torch.zeros(k, n, device="cuda")
    x[at, torch.arange(n, device="cuda")] = 1
    y = torch.empty(m, n, device="cuda")
    C.launch_count(reset=True)
    C.spmm_fwd(w, x, y, ws)
    assert C.launch_count() == 2, "a shape of the tensor-core path"
    assert torch.equal(y, dense[:, at])
    f = torch.randn(n, device="cuda", generator=_gen(7))
    C.spmm_fwd(w, x * f, y, ws)
    ref = dense[:, at].double() * f.double()
    assert bool(((y.double() - ref).abs() <= 2 * U * ref.abs()).all())


@pytest.mark.parametrize("rows,cols,n,most", [(4096, 9216, 256, 64), (4096, 4096, 1024, 72), (8192, 16384, 1024, 192)])
def test_workspace_follows_the_operands(C, rows, cols, n, most):
    """The workspace (megabytes) holds parts of X and sums, not copies of W for a matrix that is full."""
    assert C.Workspace(rows, cols, n).nbytes <= most * 1e6


def test_gradient_with_a_bad_sample_costs_a_float32_product(C):
    """One sample of infinities marks every row: right, and at the price of the CUDA-core gradient (8 times the tensor
    cores', measured) and not that of a serial sum per entry (350 times)."""
    m = k = 4096
    n = 256
    ws = C.Workspace(m, k, n)
    dy, x = torch.randn(m, n, device="cuda", generator=_gen(1)), torch.randn(k, n, device="cuda", generator=_gen(2))
    x = x.abs()
    g = torch.empty(m, k, device="cuda")
    plain = _us(lambda: C.weight_grad_dense(dy, x, g, ws, precision=0))
    dy[5:, 3] = float("inf")
    assert _us(lambda: C.weight_grad_dense(dy, x, g, ws, precision=0)) < 25 * plain
    assert bool((g[5:] == float("inf")).all())
    ref, mag = dy[:5].double() @ x.double().T, dy[:5].double().abs() @ x.double().T
    assert bool(((g[:5].double() - ref).abs() <= n * U * mag).all())
    assert ws.status()[0] == 0


@pytest.mark.parametrize("m,k,n", [(300, 520, 250), (257, 1027, 200), (64, 4096, 1024)])
def test_gradient_of_marked_operands_is_the_chain(C, m, k, n):
    """With a value that the tensor cores can't take, every entry is the float32 chain of the CUDA-core kernel, bit for
    bit (which runs without a workspace)."""
    ws = C.Workspace(m, k, n)
    dy, x = torch.randn(m, n, device="cuda", generator=_gen(m)), torch.randn(k, n, device="cuda", generator=_gen(k))
    dy[m - 1, n - 1] = 2.0 ** 100
    g, want = torch.full((m, k), float("nan"), device="cuda"), torch.full((m, k), float("nan"), device="cuda")
    C.launch_count(reset=True)
    C.weight_grad_dense(dy, x, g, ws, precision=0)
    assert C.launch_count() == 2, "a shape of the tensor-core path"
    ws.nbytes = 256     # no room for the parts
    if n <= 512:        # (longer sums over few outputs need the workspace, and are added in slices)
        C.weight_grad_dense(dy, x, want, ws, precision=0)
        assert torch.equal(_bits(g), _bits(want))
    ref, mag = dy.double() @ x.double().T, dy.double().abs() @ x.double().abs().T
    assert bool(((g.double() - ref).abs() <= n * U * mag).all())


@pytest.mark.parametrize("m,k,n", [(300, 520, 250), (513, 1027, 600), (4096, 4096, 256)])
@pytest.mark.parametrize("what", ["tiny", "samples", "large"])
def test_gradient_of_any_range(C, m, k, n, what):
    """Values down to float32's least against large ones, samples of very different scale, values up to 2^28: within
    float32's summation bound for the terms of each entry."""
    ws = C.Workspace(m, k, n)
    dy, x = torch.randn(m, n, device="cuda", generator=_gen(1)), torch.randn(k, n, device="cuda", generator=_gen(2))
    if what == "tiny":
        dy, x = dy * 2.0 ** -122, x * 2.0 ** 25
    elif what == "samples":
        dy = dy * _uniform(3, -30, 0, 1, n)
    else:
        x = x * 2.0 ** 25
    g = torch.full((m, k), float("nan"), device="cuda")
    C.launch_count(reset=True)
    C.weight_grad_dense(dy, x, g, ws, precision=0)
    assert C.launch_count() == 2, "a shape of the tensor-core path"
    ref, mag = dy.double() @ x.double().T, dy.double().abs() @ x.double().abs().T
    # the truncated steps of 64 columns (8 U), the alignment of their products (8 U), the sums' roundings, the parts left out
    lim = (n // 64 + 20) * U * mag + 2.0 ** -149
    assert bool(((g.double() - ref).abs() <= lim).all())
    assert ws.status()[0] == 0


@pytest.mark.parametrize("m,k,n", [(300, 520, 250), (2000, 1030, 97)])
def test_gradient_of_one_sample(C, m, k, n):
    """A batch of which one sample counts (the others' errors are zero): one rounding of each product and the parts that
    are left out, at most 2^-24 of it each."""
    ws = C.Workspace(m, k, n)
    dy, x = torch.zeros(m, n, device="cuda"), torch.randn(k, n, device="cuda", generator=_gen(2))
    dy[:, n // 2] = torch.randn(m, device="cuda", generator=_gen(1))
    g = torch.full((m, k), float("nan"), device="cuda")
    C.launch_count(reset=True)
    C.weight_grad_dense(dy, x, g, ws, precision=0)
    assert C.launch_count() == 2, "a shape of the tensor-core path"
    ref = dy.double() @ x.double().T
    assert bool(((g.double() - ref).abs() <= 2 * U * ref.abs()).all())


@pytest.mark.parametrize("n", [1, 3, 4, 16, 33, 66, 127, 128, 129, 255, 256, 257, 300, 512, 1023, 1024])
def test_sddmm_of_any_number_of_units(C, n):
    """The gradient at the stored entries does not depend on how many units the entries are cut into: the same bits for
    a capacity of the entries alone (a unit each) and of the dense matrix (all the GPU holds)."""
    m, k = 37, 3000
    dense = _weights(m, k, 0.005, n)
    dense[[0, 5, 6, m - 1]] = 0
    dense[9, :700] = 1
    dy, x = torch.randn(m, n, device="cuda", generator=_gen(1)), torch.randn(k, n, device="cuda", generator=_gen(2))
    ws, nnz = C.Workspace(m, k, n), int((dense != 0).sum())
    got = []
    for capacity in (nnz, m * k):
        g = torch.full((nnz + 5,), 7.0, device="cuda")
        C.weight_grad_sddmm(_csr(C, dense, ws, capacity=capacity), dy, x, g, ws)
        assert bool((g[nnz:] == 7).all())
        got.append(g[:nnz])
    assert torch.equal(_bits(got[0]), _bits(got[1]))
