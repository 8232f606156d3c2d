"""Calls beside other work: several solvers on streams and threads of their own, and a
call behind a join of two streams, eager and captured.  A call's first kernel may be
prepared while the kernel before it runs, so everything it reads has to have been
waited for."""
import threading

import pytest

import workloads as wl

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ft():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    import paper_2605_08523_gb300 as ft
    return ft


def solver(ft, n, mode, flags):
    H = torch.from_numpy(wl.chain_1d(n, n).ravel().copy()).cuda()
    s = ft.Solver([n], [0.1], [0.15], ft.ModelSet(), mode=mode, want=3, flags=flags)
    assert s.run(H, sync=True) == 0
    return H, s, (s.D.clone(), s.S.clone(), s.trace.clone())


def check(s, ref):
    assert torch.equal(s.D, ref[0]) and torch.equal(s.S, ref[1]) and torch.equal(s.trace, ref[2])


def test_solvers_on_streams_and_threads(ft):
    runs = [solver(ft, n, m, f) for n, m, f in (
        (300, "fp16x2", 0), (1024, "bf16x3", 0), (2200, "fp16x2", 0), (700, "fp32", ft.LANCZOS),
        (129, "tf32x3", ft.LANCZOS), (1600, "tf32x3", ft.REFINE2), (2600, "fp16x2", ft.EPI_DEFERRED))]
    streams = [torch.cuda.Stream() for _ in runs]
    for _, s, _ in runs:
        s.D.zero_()
    torch.cuda.synchronize()

    def work(i):
        with torch.cuda.stream(streams[i]):
            for _ in range(6):
                runs[i][1].run(runs[i][0])

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(runs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    for _, s, ref in runs:
        check(s, ref)


@pytest.mark.parametrize("flags", ["", "lanczos", "layers"])
def test_call_behind_a_join(ft, flags):
    H, s, ref = solver(ft, 300, "fp16x2", {"": 0, "lanczos": ft.LANCZOS, "layers": ft.LAYER_LAUNCHES}[flags])
    buf, main, side = torch.zeros_like(H), torch.cuda.Stream(), torch.cuda.Stream()

    def body():
        # H arrives through `side`; `main` has a kernel of its own before the join
        side.wait_stream(main)
        with torch.cuda.stream(side):
            t = H * 1.0
            for _ in range(40):
                t = t * 1.0 + 0.0
            buf.copy_(t)
        H + 1.0
        main.wait_stream(side)
        s.run(buf)
        return s.D * 2.0

    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g, stream=main):
        captured = body()
    for eager in (False, True):
        for _ in range(5):
            buf.zero_()
            s.D.zero_()
            torch.cuda.synchronize()
            if eager:
                with torch.cuda.stream(main):
                    out = body()
            else:
                g.replay()
                out = captured
            torch.cuda.synchronize()
            check(s, ref)
            assert torch.equal(out, ref[0] * 2.0)
