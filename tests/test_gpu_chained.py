"""Region calls whose launches may be scheduled while the launch before them
drains (programmatic stream serialization): each call reads what the one before
wrote, so a chain of identity regions hands the values through unchanged, also
between other work of the stream and as a captured graph."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def H():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2308_16877_gb300 import hpac
    hpac.load()
    return hpac


def chain(H, n, stream, length=24):
    """Buffers and a call that hands buffer 0 on to the last one: exact, TAF and
    iACT at threshold 0 (nothing is approximated) and perforation that drops
    nothing, in turn."""
    bufs = [torch.zeros(1, n, device="cuda") for _ in range(length + 1)]
    regs = [H.Region(H.HPAC_REGION_IDENTITY, b, logical_threads=max(1, n // 3), stream=stream) for b in bufs[:-1]]

    def run():
        for j, R in enumerate(regs):
            x, y = bufs[j], bufs[j + 1].view(-1)
            if j % 4 == 0:
                R.run_exact(x, y)
            elif j % 4 == 1:
                R.run_taf(x, y, 2, 2, 0.0, j % 3)
            elif j % 4 == 2:
                R.run_iact(x, y, 2, 4, 0.0, j % 3)
            else:
                R.run_perfo(x, y, H.HPAC_PERFO_INI, 0)
    return bufs, regs, run


@pytest.mark.parametrize("n", [97, 50001, 1 << 21])
def test_chain_on_a_stream(H, n):
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        bufs, regs, run = chain(H, n, s)
        for rep in range(8):
            src = torch.rand(1, n, device="cuda")
            for b in bufs[1:]:
                b.fill_(-1.0)
            bufs[0].copy_(src)
            run()
            out = bufs[-1] + 0.0          # another kernel of the stream reads the result
            bufs[0].zero_()               # and the first input changes behind the chain
            s.synchronize()
            assert torch.equal(out, src), rep
        for R in regs:
            R.close()


@pytest.mark.parametrize("n", [97, 1 << 20])
def test_chain_in_a_captured_graph(H, n):
    s = torch.cuda.Stream()
    src = torch.zeros(1, n, device="cuda")
    with torch.cuda.stream(s):
        bufs, regs, run = chain(H, n, s)
        run()                             # loads every kernel before the capture
        s.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            bufs[0].copy_(src)
            run()
            out = bufs[-1] + 0.0
    for rep in range(4):
        src.copy_(torch.rand(1, n, device="cuda"))
        torch.cuda.synchronize()
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, src), rep
    for R in regs:
        R.close()
