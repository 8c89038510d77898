"""tursca_csr_solve_noalloc on matrices whose rows differ a lot, where the
one-launch form cuts long rows into chunks: one row of every column, long rows
that start, end and fill a block's share, more chunks than a block lists,
lengths on either side of a chunk, with and without a window of columns.

Tolerance and reference: as in test_gpu_csr_launch.py, with the FP64 rounding
of a row of N terms, N 2^-53 of the sum of their magnitudes (at most 0.5 max|x|):
1e-11 covers the longest row here, 65,536 terms, and 1 / (1 - 0.5).
"""
import pytest

from paper_2503_16037_gb300 import tursca as T

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

CASES = {  # rows, entries of a common row (0 .. 2 k), reach of the columns (0: anywhere), long rows
    "every_column": (65536, 20, 2000, {30000: 65536}),
    "first_and_last": (3000, 10, 400, {0: 5000, 2999: 7000}),
    "chunk_edges": (20000, 30, 1000, {100 * i: n for i, n in enumerate([511, 512, 513, 1023, 1024, 1025, 4095, 4097])}),
    "more_than_a_list": (4000, 2, 300, {i: 20000 for i in range(200, 230)}),
    "many": (20000, 8, 0, {7 * i: 600 + i for i in range(1500)}),
    "long_and_wide": (2000, 400, 0, {5: 30000, 1000: 9000}),
    "no_window": (100000, 10, 0, {10000 * i: 4000 for i in range(10)}),
}


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2503_16037_gb300 import build
    build.build()


def system(name):
    n, k, reach, longs = CASES[name]
    g = torch.Generator().manual_seed(n + k)
    length = torch.randint(0, 2 * k + 1, (n,), generator=g)
    for i, m in longs.items():
        length[i] = m
    row_ptr = torch.zeros(n + 1, dtype=torch.int64)
    row_ptr[1:] = length.cumsum(0)
    nnz = int(row_ptr[-1])
    rows = torch.repeat_interleave(torch.arange(n), length)
    if reach:
        col = (rows + torch.randint(-reach, reach + 1, (nnz,), generator=g)) % n
    else:
        col = torch.randint(0, n, (nnz,), generator=g)
    val = torch.rand(nnz, generator=g) * (0.5 / length.clamp(min=1)[rows]).float()
    return n, row_ptr.int().cuda(), col.int().cuda(), val.cuda(), torch.rand(n, generator=g).cuda(), rows.cuda()


@pytest.mark.parametrize("name", list(CASES))
def test_long_rows(name):
    n, row_ptr, col, val, s, rows = system(name)
    out = []
    for _ in range(2):
        x = torch.full((n,), float("nan"), dtype=torch.float64, device="cuda")
        r2 = torch.full((1,), -1.0, dtype=torch.float64, device="cuda")
        T.tursca_csr_solve_noalloc(row_ptr, col, val, n, s, x, 24, 5, r2, torch.cuda.current_stream().cuda_stream)
        out.append((x, r2))
    ref = s.double()
    for _ in range(60):
        ref = s.double().index_add(0, rows, val.double() * ref[col.long()])
    x, r2 = out[0]
    assert float((x - ref).abs().max()) <= 1e-11 * float(ref.abs().max())
    assert 0.0 <= float(r2) <= (1e-11 * float(s.double().norm())) ** 2
    assert torch.equal(x, out[1][0]) and torch.equal(r2, out[1][1])  # sums run in a fixed order


@pytest.mark.parametrize("name", ["every_column", "many", "no_window"])
def test_a_long_row_does_not_hold_up_the_solve(name):
    """The same matrix with empty rows added up to 131,073 takes a launch per
    sweep, a warp per row: the one launch is no slower (it was two to five
    times as slow where the lanes of a common row took a long one)."""
    n, row_ptr, col, val, s, _ = system(name)
    stream = torch.cuda.current_stream().cuda_stream

    def ms(rows):
        ptr = torch.cat([row_ptr, row_ptr[-1:].expand(rows - n)])
        src = torch.cat([s, torch.ones(rows - n, device="cuda")])
        x = torch.empty(rows, dtype=torch.float64, device="cuda")
        best = float("inf")
        for _ in range(6):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            T.tursca_csr_solve_noalloc(ptr, col, val, rows, src, x, 20, 2, None, stream)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        return best

    one, per_sweep = ms(n), ms(131073)
    print("%s: one launch %.3f ms, a launch per sweep %.3f ms" % (name, one, per_sweep))
    assert one <= per_sweep
