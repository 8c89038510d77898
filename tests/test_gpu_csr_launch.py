"""tursca_csr_solve_noalloc where its one-launch form can go wrong: fewer rows
than blocks, empty rows, rows of more than 256 entries, bands that wrap around,
columns too far apart for a block's window, rows past what a block keeps, and
either side of the size where it goes back to a launch per sweep.

Tolerance: rows sum to at most 0.5, so 24 sweeps leave 2^-25 < 1e-7 of the
error, which is FP32's own level, and five refinements leave less than 1e-30:
FP64 rounding of the residual over the longest row (2000 terms, 2e-13) and
1 / (1 - 0.5) give 4e-13 of max|x|.
"""
import pytest

from paper_2503_16037_gb300 import tursca as T

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

CASES = {  # rows, entries per row (0 .. 2 k), reach of the columns (0: anywhere)
    "one_row": (1, 1, 0),
    "fewer_rows_than_blocks": (100, 8, 0),
    "wrapping_band": (5000, 20, 700),
    "anywhere": (40000, 12, 0),
    "double_window_too_large": (60000, 30, 9000),
    "long_rows": (3000, 1000, 0),
    "short_rows": (131072, 3, 2000),
    "launch_per_sweep": (131073, 3, 2000),
}


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2503_16037_gb300 import build
    build.build()


@pytest.mark.parametrize("name", list(CASES))
def test_one_launch_csr_solve(name):
    n, k, reach = CASES[name]
    g = torch.Generator().manual_seed(n)
    length = torch.randint(0, 2 * k + 1, (n,), generator=g)
    row_ptr = torch.zeros(n + 1, dtype=torch.int64)
    row_ptr[1:] = length.cumsum(0)
    nnz = int(row_ptr[-1])
    rows = torch.repeat_interleave(torch.arange(n), length)
    if reach:
        col = (rows + torch.randint(-reach, reach + 1, (nnz,), generator=g)) % n
    else:
        col = torch.randint(0, n, (nnz,), generator=g)
    val = torch.rand(nnz, generator=g) * (0.5 / length.clamp(min=1)[rows]).float()
    s = torch.rand(n, generator=g)
    dev = "cuda"
    x = torch.full((n,), float("nan"), dtype=torch.float64, device=dev)
    r2 = torch.full((1,), -1.0, dtype=torch.float64, device=dev)
    T.tursca_csr_solve_noalloc(row_ptr.int().to(dev), col.int().to(dev), val.to(dev), n, s.to(dev), x, 24, 5, r2,
                               torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    A = torch.sparse_coo_tensor(torch.stack([rows, col]), val.double(), (n, n)).coalesce()
    ref = s.double()
    for _ in range(60):  # 2^-60
        ref = s.double() + torch.mv(A, ref)
    assert float((x.cpu() - ref).abs().max()) <= 4e-13 * float(ref.abs().max())
    # the residual before the last correction
    assert 0.0 <= float(r2.item()) <= (1e-12 * float(s.double().norm())) ** 2
