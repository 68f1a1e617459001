"""Chain counts of untuned solves by pixels and by groups of one size and window,
as gfdeconv_tune_get reports them for the last solve, and a file's count, which
wins."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1609_01839_gb300 as gfd  # noqa: E402

DEV = torch.device("cuda:0")


def solve(c, M, N, n, windows):
    g = torch.Generator(device=DEV)
    g.manual_seed(1)
    y = torch.rand(M, N, generator=g, device=DEV)
    h = torch.full((3, 3), 1.0 / 9.0, device=DEV)
    u = [torch.empty_like(y) for _ in range(n)]
    c.solve_batched([{"y": y, "h": h, "sigma": 0.05, "w": windows[i % len(windows)], "eps": 1e-3,
                      "u": u[i]} for i in range(n)], 1)
    torch.cuda.synchronize()
    return c.tune_get(M, N)[3]


@pytest.mark.parametrize("M,N,n,windows,chains", [
    (256, 256, 255, (5,), 4), (256, 256, 256, (5,), 2), (256, 256, 256, (5, 7), 3),
    (1024, 1024, 63, (5,), 2), (1024, 1024, 63, (5, 9), 3), (1024, 1024, 64, (5,), 2),
    (2048, 2048, 16, (5,), 1), (2048, 2048, 16, (5, 7), 2)])
def test_untuned(M, N, n, windows, chains):
    with gfd.Context(0) as c:
        assert c.tune_get(M, N)[3] == 4
        assert solve(c, M, N, n, windows) == chains


def test_from_a_file(tmp_path):
    path = tmp_path / "t.txt"
    path.write_text("chains 3\n")
    with gfd.Context(0, tune_cache=str(path)) as c:
        assert solve(c, 64, 64, 4, (5,)) == 3
