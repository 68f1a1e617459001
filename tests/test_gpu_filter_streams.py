"""Filter calls in flight on more streams than a context has scratch sets: every
result is the one that the call gives alone (the same kernels on the same
inputs: the same bits), then and in later calls."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1609_01839_gb300 as gfd  # noqa: E402

DEV = torch.device("cuda:0")


def planes(seed, M, N):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    scale = 10.0 ** (seed % 5 - 2)  # other sizes of values: other grids of the split sums
    return [scale * torch.rand(M, N, generator=g, device=DEV) for _ in range(2)]


def test_more_streams_than_scratch_sets():
    sizes = [(2048, 1024), (64, 64), (512, 512), (8, 16), (1024, 2048), (256, 256)]
    inputs = [planes(i, *sizes[i % len(sizes)]) for i in range(20)]
    with gfd.Context(0) as c:
        alone = []
        for I, p in inputs:
            alone.append(c.guidfilter(I, p, 5, 1e-3))
            torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in inputs]
    with gfd.Context(0) as c:
        outs = [torch.empty_like(I) for I, _ in inputs]
        torch.cuda.synchronize()
        for _ in range(10):
            for (I, p), s, o in zip(inputs, streams, outs):
                c.guidfilter(I, p, 5, 1e-3, stream=s, out=o)
        torch.cuda.synchronize()
        assert all(torch.equal(a, o) for a, o in zip(alone, outs))
        for (I, p), a in zip(inputs, alone):
            assert torch.equal(a, c.guidfilter(I, p, 5, 1e-3))


def test_captured_by_the_caller():
    I, p = planes(3, 128, 256)
    with gfd.Context(0) as c:
        alone = c.guidfilter(I, p, 7, 1e-3)
        out = torch.zeros_like(I)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            c.guidfilter(I, p, 7, 1e-3, out=out)
        for _ in range(3):
            out.zero_()
            g.replay()
            assert torch.equal(alone, c.guidfilter(I, p, 7, 1e-3))
            torch.cuda.synchronize()
            assert torch.equal(alone, out)


def test_transform_beside_a_filter_call():
    """The inverse transform leaves the filter's bound of |I|, |p| alone."""
    I, p = planes(2, 512, 512)
    big = 1e9 * torch.rand(64, 64, device=DEV)
    other = torch.cuda.Stream()
    with gfd.Context(0) as c:
        alone = c.guidfilter(I, p, 5, 1e-3)
        X, x, out = c.fft2_r2c(big), torch.empty_like(big), torch.empty_like(I)
        torch.cuda.synchronize()

        def inverse():  # into a buffer of its own: the other stream writes it
            assert gfd.lib.gfdeconv_fft2_c2r(c._h, X.data_ptr(), 64, 64, x.data_ptr(),
                                             other.cuda_stream) == 0
        for _ in range(100):
            inverse()
            c.guidfilter(I, p, 5, 1e-3, out=out)
            inverse()
            assert torch.equal(alone, out)
        torch.cuda.synchronize()


@pytest.mark.parametrize("branches", [1, 2])
def test_captured_calls_at_once(branches):
    """Graphs of the caller's with a filter call in each branch, replayed on streams
    of their own: up to eight captured calls of a context may be in flight."""
    inputs = [planes(i, *((1024, 2048), (512, 512))[i % 2]) for i in range(8)]
    streams = [torch.cuda.Stream() for _ in range(8 // branches)]
    with gfd.Context(0) as c:
        alone = [c.guidfilter(I, p, 5, 1e-3) for I, p in inputs]
        outs = [torch.empty_like(I) for I, _ in inputs]
        torch.cuda.synchronize()
        graphs = []
        for q in range(len(streams)):
            g, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
            with torch.cuda.graph(g):
                main = torch.cuda.current_stream()
                side.wait_stream(main)
                for k, s in zip(range(branches), (main, side)):
                    i = q * branches + k
                    c.guidfilter(*inputs[i], 5, 1e-3, stream=s, out=outs[i])
                main.wait_stream(side)
            graphs.append(g)
        for _ in range(20):
            for o in outs:
                o.zero_()
            torch.cuda.synchronize()
            for g, s in zip(graphs, streams):
                with torch.cuda.stream(s):
                    g.replay()
            torch.cuda.synchronize()
            assert all(torch.equal(a, o) for a, o in zip(alone, outs))
