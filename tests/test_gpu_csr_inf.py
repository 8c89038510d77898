"""tursca_csr_solve_noalloc with an infinite source: the rows that gather it are
infinite, no row becomes NaN by it (rows are padded to whole quads inside, and
padding must not gather it), and the others keep their values, as with a launch
per sweep."""
import pytest

from paper_2503_16037_gb300 import tursca as T

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2503_16037_gb300 import build
    build.build()


@pytest.mark.parametrize("length", [1, 2, 3, 4, 5, 7, 8])
def test_infinite_source(length):
    n, hot = 600, 77
    g = torch.Generator().manual_seed(length)
    col = torch.randint(100, n, (n, length), generator=g)
    col[::3, -1] = hot  # every third row's last entry
    val = 0.1 + torch.rand(n, length, generator=g) * (0.4 / length)
    s = torch.rand(n, generator=g)
    s[hot] = float("inf")
    ptr = torch.arange(n + 1, dtype=torch.int32) * length
    x = torch.zeros(n, dtype=torch.float64, device="cuda")
    T.tursca_csr_solve_noalloc(ptr.cuda(), col.int().reshape(-1).contiguous().cuda(), val.reshape(-1).contiguous().cuda(),
                               n, s.cuda(), x, 1, 1, None, torch.cuda.current_stream().cuda_stream)
    ref = s + (val * s[col]).sum(1)  # one sweep
    x = x.cpu()
    assert torch.equal(torch.isinf(ref), torch.isinf(x)) and not bool(torch.isnan(x).any())
    fin = torch.isfinite(ref)
    # FP32 sums of at most 9 terms: 9 * 2^-24 of their magnitudes
    assert bool(((x - ref.double()).abs()[fin] <= 6e-7 * ref.double().abs()[fin]).all())
