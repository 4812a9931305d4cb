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


FIRST_QUALITY_CALL = """
import ctypes, threading
import torch
from paper_2308_16877_gb300 import hpac
hpac.load()
a = torch.rand(5000, dtype=torch.float64, device="cuda") + 0.5
b = a.float()
other = torch.cuda.Stream()
torch.cuda.synchronize()
cu = ctypes.CDLL("libcuda.so.1")
st, graph = ctypes.c_void_p(), ctypes.c_void_p()
assert cu.cuStreamCreate(ctypes.byref(st), 0) == 0            # a blocking stream
assert cu.cuStreamBeginCapture_v2(st, 1) == 0                 # thread-local mode
got = []
def work():
    with torch.cuda.stream(other):
        got.append(hpac.quality(a, b, hpac.HPAC_METRIC_RMSE))
t = threading.Thread(target=work)
t.start()
t.join()
assert cu.cuStreamEndCapture(st, ctypes.byref(graph)) == 0, "capture broken"
assert got and 0 < got[0]["value"] < 1e-6, got
print("ok")
"""


def test_first_quality_call_beside_a_capture():
    """The first hpac_quality call of a process sets up its scratch; a capture of
    a blocking stream on another thread stays valid, and the call succeeds."""
    import os
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", FIRST_QUALITY_CALL], cwd=root, capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout + r.stderr
