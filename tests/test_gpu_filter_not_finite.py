"""A pixel that is not finite in a call of the guided filter: outputs more than w + 5
pixels away (2 r = w - 1 by the windows, up to 3 more along a row and 3 down a
column in either stage, where sums of a lane's four columns and of four rows are
slid) are those of a finite pixel in its place.  Tolerance 1e-5 of the values' size: what
plain FP32 sums would reach (2^-24 times some tens of additions, over eps +
variance of order 0.1)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1609_01839_gb300 as gfd  # noqa: E402

DEV = torch.device("cuda:0")


@pytest.mark.parametrize("mode", [gfd.VAR_COMPENSATED, gfd.VAR_FP64, gfd.VAR_DOUBLE_FLOAT])
@pytest.mark.parametrize("value", [np.nan, np.inf])
@pytest.mark.parametrize("plane", [0, 1])
def test_stays_where_it_is(mode, value, plane):
    M, N, w = 1024, 2048, 5
    g = torch.Generator(device=DEV)
    g.manual_seed(9)
    planes = [torch.rand(M, N, generator=g, device=DEV) for _ in range(2)]
    ii, jj = torch.arange(M, device=DEV)[:, None], torch.arange(N, device=DEV)[None, :]
    with gfd.Context(0, var_precision=mode) as c:
        want = c.guidfilter(*planes, w, 0.1)
        far = torch.ones(M, N, dtype=torch.bool, device=DEV)
        bad = [x.clone() for x in planes]
        for y in range(0, M, 97):  # every row of an item, centres of items among them
            for x in (y % 128, 60 + y, 1500 + y // 8):
                bad[plane][y, x % N] = value
                dy, dx = (ii - y).abs(), (jj - x % N).abs()
                far &= ~((torch.minimum(dy, M - dy) <= w + 5) & (torch.minimum(dx, N - dx) <= w + 5))
        got = c.guidfilter(*bad, w, 0.1)
    assert float(far.float().mean()) > 0.9
    assert float((got - want).abs()[far].max()) < 1e-5  # (false for NaN)
    assert not bool(torch.isfinite(got[~torch.isfinite(bad[plane])]).any())


@pytest.mark.parametrize("mode", [gfd.VAR_COMPENSATED, gfd.VAR_FP64, gfd.VAR_DOUBLE_FLOAT])
def test_at_every_place_of_an_item(mode):
    """The centre of an item is its reference: no place may matter."""
    M = N = 128
    g = torch.Generator(device=DEV)
    g.manual_seed(10)
    I, p = (torch.rand(M, N, generator=g, device=DEV) for _ in range(2))
    with gfd.Context(0, var_precision=mode) as c:
        want = c.guidfilter(I, p, 3, 0.1)
        for y in range(0, M, 5):
            for x in (0, 1, 59, 60, 61, 62, 127):
                J = I.clone()
                J[y, x] = float("nan")
                got = c.guidfilter(J, p, 3, 0.1)
                dy = (torch.arange(M, device=DEV)[:, None] - y).abs()
                dx = (torch.arange(N, device=DEV)[None, :] - x).abs()
                far = ~((torch.minimum(dy, M - dy) <= 8) & (torch.minimum(dx, N - dx) <= 8))
                assert float((got - want).abs()[far].max()) < 1e-5, (y, x)


@pytest.mark.parametrize("boundary", [gfd.BOUNDARY_PERIODIC, gfd.BOUNDARY_TRUNCATED])
def test_infinite_pixels_leave_the_grid(boundary):
    """The grid of the split sums rests on the finite pixels: away from infinite ones
    the sums are as good as without them.  Nearly flat planes much smaller than one, eps
    far below what plain FP32 sums of the deviations resolve; measured against FP64
    sums, with room for the sums that are formed again from the ring of rows."""
    M, N, w = 256, 512, 9
    g = torch.Generator(device=DEV)
    g.manual_seed(12)
    ramp = torch.linspace(0.0, 0.1, M, device=DEV)[:, None] * torch.ones(M, N, device=DEV)
    I, p = (ramp + 1e-3 * torch.rand(M, N, generator=g, device=DEV) for _ in range(2))
    J, q = I.clone(), p.clone()
    J[100, 200], q[180, 400] = float("inf"), float("-inf")
    dy = torch.arange(M, device=DEV)[:, None]
    dx = torch.arange(N, device=DEV)[None, :]
    far = torch.ones(M, N, dtype=torch.bool, device=DEV)
    for y, x in ((100, 200), (180, 400)):
        far &= ((dy - y).abs() > w + 5) | ((dx - x).abs() > w + 5)
    with gfd.Context(0, var_precision=gfd.VAR_FP64, boundary=boundary) as c:
        want = c.guidfilter(I, p, w, 1e-7)
    with gfd.Context(0, boundary=boundary) as c:
        alone = (c.guidfilter(I, p, w, 1e-7) - want).abs()[far].max()
        beside = (c.guidfilter(J, q, w, 1e-7) - want).abs()[far].max()
    assert float(beside) <= 4 * float(alone)
